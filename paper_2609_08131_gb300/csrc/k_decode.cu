// k_decode.cu - the pieces of decoding-stage eviction that the prefill pass
// does not already have.
//
// During decoding the query statistics are estimated from the queries seen so
// far (Sec. 3.4, last paragraph), not from a fixed window: every decode step
// adds one query per (request, layer, query head). The running statistics are
// kept as (count n, mean m, sum of squared deviations M2) per channel and a
// batch of new queries is merged with the pairwise update of Chan, Golub and
// LeVeque (1979):
//   n = n_a + n_b,  delta = m_b - m_a,  m = m_a + delta n_b / n,
//   M2 = M2_a + M2_b + delta^2 n_a n_b / n,
// with (m_b, M2_b) of the batch taken in two passes. At an eviction the
// scoring pass reads mu = m and lambda = M2 / n (or M2 / (n - 1)) instead of
// window statistics.
//
// After the TOP-B selection the cache of a request is compacted in place so
// that the kept rows occupy rows 0 .. kept - 1 of the request's range, in one
// of two ways (one CTA per unit in both; jacap_inplace.cuh holds the per-unit
// code, which the selection kernel also runs right after selecting a unit):
//  - ascending order (the order of jacap_compact): every kept row moves to
//    its rank. The rows move in chunks; every chunk is read completely before
//    any of it is written (a barrier in between). Because the kept positions
//    ascend strictly from 0, idx[r] >= r, so a chunk's writes (rows c0 ..
//    c0 + CH - 1) never touch a row that a later chunk still has to read
//    (rows >= c0 + CH). Up to `kept` rows move.
//  - hole filling: kept rows below `kept` stay where they are; the kept rows
//    at or above `kept` move, in ascending order, into the evicted rows below
//    `kept`, in ascending order. Sources and destinations are disjoint, so all
//    copies run at once, and at most n - kept rows move (the eviction interval
//    during decoding, instead of the whole budget). If f kept positions lie
//    below `kept`, the evicted row r between the (i-1)-th and i-th of them is
//    hole number r - i and receives row idx[f + r - i].
#include "jacap_dev.cuh"
#include "jacap_inplace.cuh"
#include "jacap_internal.h"

namespace jacap {

template <typename T>
__device__ __forceinline__ float q_elem(const T* p);
template <>
__device__ __forceinline__ float q_elem<float>(const float* p) { return __ldg(p); }
template <>
__device__ __forceinline__ float q_elem<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// One block per (request, layer, query head); thread c owns channel c.
// stats: [S][L][Hq][2][D] (mean, M2); counts: [S][L][Hq].
template <typename T>
__global__ void __launch_bounds__(D)
    stats_update_kernel(Dims dm, const T* __restrict__ q, float* stats, int32_t* counts, int reset) {
  pdl_wait();
  const int b = blockIdx.x;
  const int h = b % dm.Hq;
  const int l = (b / dm.Hq) % dm.L;
  const int s = b / (dm.Hq * dm.L);
  const int c = threadIdx.x;
  const T* base = q + (int64_t)s * dm.q_ss + (int64_t)l * dm.q_sl + (int64_t)h * dm.q_sh + c;
  const int nb = dm.window;
  float sum = 0.f;
  for (int j = 0; j < nb; ++j) sum += q_elem(base + (int64_t)j * dm.q_sp);
  const float mb = sum / (float)nb;
  float m2b = 0.f;
  for (int j = 0; j < nb; ++j) {
    const float e = q_elem(base + (int64_t)j * dm.q_sp) - mb;
    m2b = fmaf(e, e, m2b);
  }
  float* st = stats + (int64_t)b * 2 * D;
  int na = reset ? 0 : counts[b];
  if (na < 0) na = 0;
  float mean = mb, m2 = m2b;
  if (na > 0) {
    const float n = (float)na + (float)nb;
    const float ma = st[c], delta = mb - ma;
    mean = fmaf(delta, (float)nb / n, ma);
    m2 = st[D + c] + m2b + delta * delta * ((float)na * (float)nb / n);
  }
  __syncthreads();  // every thread has read counts[b] before it changes
  st[c] = mean;
  st[D + c] = m2;
  if (c == 0) counts[b] = na + nb;
}

// One decode step of up to AP_MAX requests: a block per (request, layer, query
// head) merges the head's query into the running statistics, one channel per thread,
// with the arithmetic of stats_update_kernel for a batch of one; the first head of a
// group's block also copies the new K and V rows (16-byte pieces) and the tag into
// the request's next free slot row. Bound: the launch and two dependent reads (4
// requests x 28 layers x 28 heads: 4 us; a block per KV head that took its seven
// heads in turn: 16 us). One launch with the rows' numbers as arguments replaces two
// index tensors copied from the host (each a synchronisation of the stream), three
// indexed copies and the update: 170 -> 20 us of host time a step, and the steps no
// longer wait for the device.
constexpr int AP_MAX = 256;
struct AppendRows {
  int32_t row[AP_MAX], id[AP_MAX];
};

template <typename T>
__global__ void __launch_bounds__(D)
    append_kernel(Dims dm, AppendArgs a, const __grid_constant__ AppendRows rows, int s0) {
  pdl_wait();
  const int b = blockIdx.x, tid = threadIdx.x;
  const int hq = b % dm.Hq, l = (b / dm.Hq) % dm.L, sl = b / (dm.Hq * dm.L), s = s0 + sl;
  const int64_t sb = ((int64_t)s * dm.L + l) * dm.Hq + hq;
  float* st = a.stats + sb * 2 * D;
  const float x = q_elem((const T*)a.q_new + s * dm.q_ss + l * dm.q_sl + hq * dm.q_sh + tid);
  const float ma = st[tid], sa = st[D + tid];
  int na = a.counts[sb];
  if (hq % dm.G == 0) {
    constexpr int CH = D * (int)sizeof(T) / 16;  // 16-byte pieces of a row
    const int g = hq / dm.G;
    const int64_t row = (int64_t)s * a.slot_rows + rows.row[sl];
    if (tid < 2 * CH) {
      const bool isv = tid >= CH;
      const int p = isv ? tid - CH : tid;
      const int64_t* str = a.strides + (isv ? 3 : 0);
      const T* src = (const T*)(isv ? a.v_new : a.k_new) + s * str[0] + l * str[1] + g * str[2];
      T* dst = (T*)(isv ? a.v : a.k) + (int64_t)l * dm.kv_sl + (int64_t)g * dm.kv_sh + row * dm.kv_st;
      ((uint4*)dst)[p] = ((const uint4*)src)[p];
    } else if (tid == 2 * CH && a.pos != nullptr) {
      a.pos[(int64_t)l * (dm.kv_sl / dm.kv_st) + (int64_t)g * (dm.kv_sh / dm.kv_st) + row] = rows.id[sl];
    }
  }
  if (na < 0) na = 0;
  float mean = x, m2 = 0.f;
  if (na > 0) {
    const float n = (float)na + 1.f;
    const float delta = x - ma;
    mean = fmaf(delta, 1.f / n, ma);
    m2 = sa + delta * delta * ((float)na / n);
  }
  __syncthreads();  // every thread has read counts before it changes
  st[tid] = mean;
  st[D + tid] = m2;
  if (tid == 0) a.counts[sb] = na + 1;
}

// The scoring pass's query statistics from running statistics: the same
// outputs as the window statistics (mu / (tau sqrt d) and lambda).
__global__ void __launch_bounds__(D)
    stats_moments_kernel(Dims dm, Ws ws, const float* __restrict__ stats, const int32_t* __restrict__ counts) {
  pdl_wait();
  if (status_failed(ws)) return;
  const int b = blockIdx.x, c = threadIdx.x;
  const int n = counts[b];
  if (n < (dm.cov_unbiased ? 2 : 1)) {
    if (c == 0) flag(ws, ST_INVALID);
    return;
  }
  const float mean = stats[(int64_t)b * 2 * D + c];
  const float lam = stats[(int64_t)b * 2 * D + D + c] / (float)(dm.cov_unbiased ? n - 1 : n);
  ws.mu[(int64_t)b * D + c] = mean * dm.inv_scale;
  ws.lam[(int64_t)b * D + c] = lam;
  if (!isfinite(mean) || !isfinite(lam) || lam < 0.f) flag(ws, ST_NONFINITE);
}

constexpr int CI_THREADS = 256;

// One CTA per unit u = (l Hkv + g) S + s, the order of jacap_select's idx. The
// kept positions come from the caller: a unit whose positions do not ascend
// strictly within [0, n) is left untouched and flagged.
template <typename T>
__global__ void __launch_bounds__(CI_THREADS)
    compact_inplace_kernel(Dims dm, Ws ws, const int32_t* __restrict__ cu, T* k, T* v, int32_t* pos,
                           const int32_t* __restrict__ idx, int budget) {
  pdl_wait();
  // together, as a block of this launch may set the word (a unit's positions)
  if (__syncthreads_or(status_failed(ws) ? 1 : 0)) return;
  const int u = blockIdx.x;
  const int s = u % dm.S, plane = u / dm.S;
  const int tid = threadIdx.x;
  const int64_t t0 = cu[s];
  const int64_t n = (int64_t)cu[s + 1] - t0;
  const int kept = (int)(n < (int64_t)budget ? n : (int64_t)budget);
  const int32_t* ix = idx + (int64_t)u * budget;
  int bad = 0;
  for (int r = tid; r < kept; r += CI_THREADS) {
    const int32_t x = ix[r];
    bad |= x < 0 || (int64_t)x >= n || (r > 0 && x <= ix[r - 1]);
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) flag(ws, ST_INVALID);
    return;
  }
  compact_ordered_unit<T, CI_THREADS>(dm, plane, t0, kept, k, v, pos, ix);
}

template <typename T>
__global__ void __launch_bounds__(CI_THREADS)
    fill_holes_kernel(Dims dm, Ws ws, const int32_t* __restrict__ cu, T* k, T* v, int32_t* pos,
                      const int32_t* __restrict__ idx, int budget) {
  pdl_wait();
  __shared__ int s_f;
  if (__syncthreads_or(status_failed(ws) ? 1 : 0)) return;  // together, as above
  const int u = blockIdx.x;
  const int s = u % dm.S, plane = u / dm.S;
  const int tid = threadIdx.x;
  const int64_t t0 = cu[s];
  const int64_t n = (int64_t)cu[s + 1] - t0;
  const int kept = (int)(n < (int64_t)budget ? n : (int64_t)budget);
  const int32_t* ix = idx + (int64_t)u * budget;
  if (tid == 0) s_f = 0;
  __syncthreads();
  int bad = 0;
  for (int r = tid; r < kept; r += CI_THREADS) {
    const int32_t x = ix[r];
    bad |= x < 0 || (int64_t)x >= n || (r > 0 && x <= ix[r - 1]);
    // f = the number of kept positions below `kept`
    if (x < kept && (r + 1 == kept || ix[r + 1] >= kept)) s_f = r + 1;
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) flag(ws, ST_INVALID);
    return;
  }
  fill_holes_unit<T, CI_THREADS>(dm, plane, t0, kept, s_f, 0, 1, k, v, pos, ix);
}

template <typename T>
static cudaError_t launch_stats_update_t(const Dims& dm, const void* q, float* stats, int32_t* counts, int reset,
                                         cudaStream_t st) {
  JACAP_TRY(launch_pdl(dm.pdl != 0, stats_update_kernel<T>, dm.S * dm.L * dm.Hq, D, 0, st, dm, (const T*)q, stats,
                       counts, reset));
  return cudaGetLastError();
}

cudaError_t launch_stats_update(const Dims& dm, int dtype, const void* q, float* stats, int32_t* counts, int reset,
                                cudaStream_t st) {
  return dtype == 1 ? launch_stats_update_t<__nv_bfloat16>(dm, q, stats, counts, reset, st)
                    : launch_stats_update_t<float>(dm, q, stats, counts, reset, st);
}

cudaError_t launch_append(const Dims& dm, int dtype, const AppendArgs& a, const int32_t* lengths, const int32_t* ids,
                          cudaStream_t st) {
  for (int s0 = 0; s0 < dm.S; s0 += AP_MAX) {
    const int n = dm.S - s0 < AP_MAX ? dm.S - s0 : AP_MAX;
    AppendRows rows;
    for (int i = 0; i < AP_MAX; ++i) {
      rows.row[i] = i < n ? lengths[s0 + i] : 0;
      rows.id[i] = i < n ? ids[s0 + i] : 0;
    }
    const int blocks = n * dm.L * dm.Hq;
    if (dtype == 1)
      JACAP_TRY(launch_pdl(dm.pdl != 0, append_kernel<__nv_bfloat16>, blocks, D, 0, st, dm, a, rows, s0));
    else
      JACAP_TRY(launch_pdl(dm.pdl != 0, append_kernel<float>, blocks, D, 0, st, dm, a, rows, s0));
  }
  return cudaGetLastError();
}

cudaError_t launch_stats_moments(const Dims& dm, const Ws& ws, const float* stats, const int32_t* counts,
                                 cudaStream_t st) {
  JACAP_TRY(launch_pdl(dm.pdl != 0, stats_moments_kernel, dm.S * dm.L * dm.Hq, D, 0, st, dm, ws, stats, counts));
  return cudaGetLastError();
}

cudaError_t launch_compact_inplace(const Dims& dm, const Ws& ws, int dtype, const int32_t* cu, void* k, void* v,
                                   int32_t* pos, const int32_t* idx, int budget, int preserve_order,
                                   cudaStream_t st) {
  const int units = dm.L * dm.Hkv * dm.S;
  if (!preserve_order) {
    if (dtype == 1)
      JACAP_TRY(launch_pdl(dm.pdl != 0, fill_holes_kernel<__nv_bfloat16>, units, CI_THREADS, 0, st, dm, ws, cu,
                           (__nv_bfloat16*)k, (__nv_bfloat16*)v, pos, idx, budget));
    else
      JACAP_TRY(launch_pdl(dm.pdl != 0, fill_holes_kernel<float>, units, CI_THREADS, 0, st, dm, ws, cu, (float*)k,
                           (float*)v, pos, idx, budget));
    return cudaGetLastError();
  }
  if (dtype == 1)
    JACAP_TRY(launch_pdl(dm.pdl != 0, compact_inplace_kernel<__nv_bfloat16>, units, CI_THREADS, 0, st, dm, ws, cu,
                         (__nv_bfloat16*)k, (__nv_bfloat16*)v, pos, idx, budget));
  else
    JACAP_TRY(launch_pdl(dm.pdl != 0, compact_inplace_kernel<float>, units, CI_THREADS, 0, st, dm, ws, cu, (float*)k,
                         (float*)v, pos, idx, budget));
  return cudaGetLastError();
}

}  // namespace jacap
