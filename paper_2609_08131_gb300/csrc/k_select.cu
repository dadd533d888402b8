// k_select.cu - TOP-B selection (Algorithm 1 step 5) and compaction of the
// retained cache Z_C (Sec. 3.1).
//
// select_kernel: one CTA per unit. Scores are non-negative float32, so their bit
// patterns order like unsigned integers. The kept set of a unit of more than B
// tokens is {key > T} and the first keys == T by position, for the key T of the
// B-th token in the order of Algorithm 1 (score descending, then position):
//  1. histogram of the keys in SE_FINE bins of 2^16 (1/128 octave each: 15.75
//     octaves, in which the lanes of a warp rarely meet in one bin) that end just
//     above the maximum (of the first slab and a sample of the others);
//  2. the bin that holds the B-th key, by a scan over all warps;
//  3. that bin's keys (a handful) go to a list, and each one's rank in it names T
//     and the number of keys == T that are kept.
// If the B-th key lies above or below the fine bins, a histogram of 2048 bins over
// the keys there names its bin. While a bin holds more than SE_CAND keys (many ties,
// as with a window of one query), a histogram over its next 11 bits names a smaller
// one. Each of these reads the keys once more, from registers where one slab holds
// them.
// Emission: the keys are held in registers in slabs of NT KPT (KPT per lane, all
// loads in flight together; the smallest that holds the longest request; a longer
// one is read again by each step, from L2); warp w owns 32 KPT consecutive
// positions, lane j keeps the ballot of slot j, and prefix sums of the counts over
// lanes and warps place each lane's positions: ascending, and deterministic.
//
// With fewer units than SMs, `parts` CTAs take a unit: each selects for itself (the
// SMs would idle otherwise; all write the same positions) and moves its share of
// the rows.
//
// Bound: latency and shared-memory atomics of one unit, then the row copies (HBM).
// Why one CTA per unit dealt by the hardware, and small CTAs for short requests:
// a resident grid that strides over the units gave a CTA the same request of a
// batch each time when the number of requests divided the grid.
// Measured against three radix passes over all keys in such a grid, selection and
// row copies: 1024 units of 731-3072 tokens (256 kept) 0.152 -> 0.055 ms, 1024 units
// of 2K-64K tokens (512) 0.290 -> 0.155, 320 units of 9001 (900) 0.102 -> 0.079, 256
// units of 32768 (512) 0.057 -> 0.043, of 131072 (1024) 0.154 -> 0.119, 8 units of
// 4099 (512) 0.018 -> 0.011; 448 slots of 2052 tokens with holes filled 0.045 -> 0.020.
// The copies' bytes alone take 0.040, 0.079, 0.044, 0.020 and 0.040 ms of the first
// five at the copy rate.
//
// compact_kernel: 16-byte vector copies of the kept K and V rows into the
// dense [L][Hkv][S][B][d] output; rows of -1 (or of a position outside the
// request) are zero-filled, so no index value can make it read out of bounds.
//
// select_kernel can also finish each unit itself as soon as its positions are
// emitted, so the rows move while other CTAs are still selecting and no
// separate compaction launch follows: MODE 1 copies the kept rows into k_out,
// v_out (the work of compact_kernel, same zero fill); MODE 2 fills the holes
// of the cache in place (jacap_inplace.cuh, as jacap_compact_inplace does).
// MODE 0 only selects. (The in-place compaction in ascending order moves
// every kept row; it stays a launch of its own, whose small CTAs keep more
// bytes in flight per SM than one selection CTA per unit could.)
#include <algorithm>

#include "jacap_dev.cuh"
#include "jacap_inplace.cuh"
#include "jacap_internal.h"

namespace jacap {


constexpr int SE_BINS = 2048;
constexpr int SE_FINE = 2016;   // bins of 2^16 keys, below bin 0 (every key above them)
constexpr int SE_CAND = 256;    // keys of the B-th key's bin that are ranked directly (a rank reads them all: ~3 us)
constexpr int SE_IDX = 2048;    // kept positions also held in shared memory

struct SeSmem {
  uint32_t hist[SE_BINS];
  __align__(16) uint32_t ckey[SE_CAND];
  __align__(16) int32_t cidx[SE_CAND];
  int32_t idx[SE_IDX];
  uint32_t tot[2][32];  // counts per warp
  uint32_t max, digit, need, count, T;
  int skip;
};

// Keys of slab `sl` into registers: lane's register j holds position
// sl * NT KPT + 32 KPT w + 32 j + lane (coalesced; all loads in flight at
// once). KPT keys per lane (4 .. 32) is chosen from the longest request, so a
// short cache does not carry empty register slots through every pass.
template <int KPT, int NT>
__device__ __forceinline__ void load_slab(const uint32_t* key, int n, int sl, int warp, int lane,
                                          uint32_t (&kr)[KPT]) {
  const int base = sl * NT * KPT + warp * (32 * KPT) + lane;
#pragma unroll
  for (int j = 0; j < KPT; ++j) {
    const int i = base + 32 * j;
    kr[j] = i < n ? __ldg(key + i) : 0u;
  }
}

// Rows out[0 .. B) of unit u (positions relative to the request start, as
// emitted; the first SE_IDX also in sidx if not null) from K and V into k_out,
// v_out; -1 or a position outside the request gives a zero row. Part `part` of
// `parts` of the copies. All threads of the CTA; out and sidx were written by them before the barrier that precedes this
// call.
template <typename T, int NT>
__device__ __forceinline__ void gather_unit(const Dims& dm, int plane, int64_t start, int64_t end, bool valid,
                                            const T* __restrict__ k, const T* __restrict__ v,
                                            const int32_t* out, const int32_t* sidx, int B, int64_t u, int part,
                                            int parts, T* __restrict__ k_out, T* __restrict__ v_out) {
  constexpr int CH = D * (int)sizeof(T) / 16;  // 16-byte chunks per row
  const int l = plane / dm.Hkv, g = plane % dm.Hkv;
  const int64_t base = (int64_t)l * dm.kv_sl + (int64_t)g * dm.kv_sh;
  uint4* ko = (uint4*)(k_out + u * B * D);
  uint4* vo = (uint4*)(v_out + u * B * D);
#pragma unroll 4
  for (int e = part * NT + threadIdx.x; e < B * CH; e += parts * NT) {
    const int r = e / CH, c = e % CH;
    const int32_t src = sidx != nullptr && r < SE_IDX ? sidx[r] : out[r];
    uint4 kk = make_uint4(0, 0, 0, 0), vv = make_uint4(0, 0, 0, 0);
    if (valid && src >= 0 && start + src < end) {
      const int64_t off = base + (start + src) * dm.kv_st;
      kk = *((const uint4*)(k + off) + c);
      vv = *((const uint4*)(v + off) + c);
    }
    ko[e] = kk;
    vo[e] = vv;
  }
}

// The digit d (0 .. SE_BINS - 1) with (sum of hist over digits before d) < need <=
// (that sum + hist[d]) into sm.digit; need less that sum into sm.need and hist[d]
// into sm.count; SE_BINS if the histogram holds fewer than `need`. Every thread of
// the CTA; the histogram is complete.
template <int NT>
__device__ __forceinline__ void find_digit(SeSmem& sm, uint32_t need, int tid) {
  constexpr int PER = SE_BINS / NT, NW = NT / 32;
  const int lane = tid & 31, warp = tid >> 5;
  uint32_t c[PER], sum = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    c[k] = sm.hist[tid * PER + k];
    sum += c[k];
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sm.tot[0][warp] = inc;
  __syncthreads();
  uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp && lane < NW ? sm.tot[0][lane] : 0u) + inc - sum;
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    if (before < need && before + c[k] >= need) {  // one thread, one k
      sm.digit = (uint32_t)(tid * PER + k);
      sm.need = need - before;
      sm.count = c[k];
    }
    before += c[k];
  }
  if (tid == NT - 1 && before < need) {
    sm.digit = SE_BINS;
    sm.need = need - before;
  }
  __syncthreads();
}

template <int KPT, typename E, int MODE, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT)
    select_kernel(Dims dm, Ws ws, const int32_t* __restrict__ cu, const float* __restrict__ scores, int B,
                  int32_t* __restrict__ idx, int32_t* __restrict__ kept, const E* __restrict__ k,
                  const E* __restrict__ v, E* __restrict__ k_out, E* __restrict__ v_out, E* kio, E* vio,
                  int32_t* pos, int parts) {
  constexpr bool GATHER = MODE == 1;
  pdl_wait();
  constexpr int SLAB = NT * KPT;  // warp w holds positions 32 KPT w .. + 32 KPT - 1 of a slab
  constexpr int NW = NT / 32;
  __shared__ SeSmem sm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int u = blockIdx.x / parts, part = blockIdx.x % parts;
  const int plane = u / dm.S, s = u % dm.S;
  const int64_t start = cu[s];
  const int64_t end = cu[s + 1];
  if (tid == 0) {
    // (not a bit that another CTA of this launch may have set)
    sm.skip = (*((volatile uint32_t*)ws.status) & ~(uint32_t)ST_SELECT) != 0u ? 1 : 0;
    sm.max = 0;
  }
  for (int b = tid; b < SE_BINS; b += NT) sm.hist[b] = 0;
  __syncthreads();
  if (sm.skip) return;
  // time accounting (trace builds, thread 0): 0 the scores loaded (one slab) and
  // their maximum, 1 the B-th token, 2 the emission, 3 the rows gathered, 4 units,
  // 5 the whole unit (units of more than B tokens)
  TRC_DECL(TR_CTA_SLOTS);
  TRC_T(tr_u);
  int32_t* out = idx + (int64_t)u * B;
  const bool valid = !(start < 0 || end < start || end > dm.Ntot);
  const int n = valid ? (int)(end - start) : 0;
  if (!valid && tid == 0) flag(ws, ST_SELECT);  // malformed cu_seqlens: no reads
  if (plane == 0 && tid == 0) kept[s] = min(n, B);
  if (n <= B) {
    for (int r = tid; r < B; r += NT) out[r] = r < n ? r : -1;
    if constexpr (GATHER) {
      __syncthreads();
      gather_unit<E, NT>(dm, plane, start, end, valid, k, v, out, nullptr, B, u, part, parts, k_out, v_out);
    }
    return;
  }
  const uint32_t* key = (const uint32_t*)(scores + (int64_t)plane * dm.Ntot + start);
  const int nslab = (n + SLAB - 1) / SLAB;
  uint32_t kr[KPT];
  TRC_INC(4);
  load_slab<KPT, NT>(key, n, 0, warp, lane, kr);  // one slab: register-resident for all steps
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < KPT; ++j) m = max(m, kr[j]);
  if (nslab > 1) {  // of the other slabs, every 16th line
#pragma unroll 8
    for (int i = SLAB + warp * 512 + lane; i < n; i += NW * 512) m = max(m, __ldg(key + i));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (lane == 0) atomicMax(&sm.max, m);
  __syncthreads();
  TRC_ADD(0, tr_u);
  TRC_T(tr_r);
  // The fine bins end above the maximum, or an octave above it if it is that of a
  // part of the keys; their ends are multiples of 2^21 keys.
  const uint32_t up = nslab > 1 ? 1u << 23 : 0u;
  const int top = (int)((min(sm.max, 0xffffffffu - up) + up) >> 16) | 31;
#pragma unroll 1
  for (int sl = 0; sl < nslab; ++sl) {
    if (sl > 0) load_slab<KPT, NT>(key, n, sl, warp, lane, kr);
    const int base = sl * SLAB + warp * (32 * KPT) + lane;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const int d = max(top - (int)(kr[j] >> 16), -1) + 1;
      if (base + 32 * j < n && d <= SE_FINE) atomicAdd(&sm.hist[d], 1u);
    }
  }
  __syncthreads();
  find_digit<NT>(sm, (uint32_t)B, tid);
  // hist[digit(key)] over the keys (SE_BINS: not counted)
  auto histogram = [&](auto digit) {
    __syncthreads();  // everyone has read digit, need and count
    for (int b = tid; b < SE_BINS; b += NT) sm.hist[b] = 0;
    __syncthreads();
#pragma unroll 1
    for (int sl = 0; sl < nslab; ++sl) {
      if (nslab > 1) load_slab<KPT, NT>(key, n, sl, warp, lane, kr);
      const int base = sl * SLAB + warp * (32 * KPT) + lane;
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        const uint32_t d = digit(kr[j]);
        if (base + 32 * j < n && d < SE_BINS) atomicAdd(&sm.hist[d], 1u);
      }
    }
    __syncthreads();
  };
  // The sm.need-th of the sm.count keys with (key >> bits) == pre is the B-th.
  uint32_t pre = (uint32_t)(top + 1 - (int)sm.digit);
  int bits = 16;
  if (sm.digit == 0 || sm.digit == SE_BINS) {
    // above or below the fine bins: the keys there by their first 11 bits; 0, which
    // many scores may be, has a bin of its own
    const bool over = sm.digit == 0;
    const uint32_t high = over ? 2047u : 2046u, left = over ? (uint32_t)B : sm.need;
    histogram([&](uint32_t x) {
      const int f = top - (int)(x >> 16);
      return (over ? f < 0 : f >= SE_FINE) ? (x == 0u ? 2047u : high - (x >> 21)) : (uint32_t)SE_BINS;
    });
    find_digit<NT>(sm, left, tid);
    bits = sm.digit == 2047u ? 0 : 21;
    pre = sm.digit == 2047u ? 0u : high - sm.digit;
  }
#pragma unroll 1
  while (sm.count > SE_CAND && bits > 0) {  // too many to rank: the next digit of those keys
    const int w = min(bits, 11);
    const uint32_t dmask = (1u << w) - 1u, left = sm.need;
    histogram([&](uint32_t x) { return x >> bits == pre ? ~(x >> (bits - w)) & dmask : (uint32_t)SE_BINS; });
    find_digit<NT>(sm, left, tid);
    pre = (pre << w) | (~sm.digit & dmask);
    bits -= w;
  }
  const int cand = (int)sm.count;
  // The B-th key T; the first sm.need of the keys == T are kept.
  uint32_t T = pre;  // (cand > SE_CAND: the whole key)
  if (cand <= SE_CAND) {
    __syncthreads();  // everyone has read the bin's count
    if (tid == 0) sm.count = 0;
    if (tid < 4 && cand + tid < SE_CAND) {  // ranked four at a time: the last ones count for nobody
      sm.ckey[cand + tid] = 0u;
      sm.cidx[cand + tid] = INT32_MAX;
    }
    __syncthreads();
#pragma unroll 1
    for (int sl = 0; sl < nslab; ++sl) {
      if (nslab > 1) load_slab<KPT, NT>(key, n, sl, warp, lane, kr);
      const int base = sl * SLAB + warp * (32 * KPT) + lane;
#pragma unroll
      for (int j = 0; j < KPT; ++j) {
        if (base + 32 * j < n && kr[j] >> bits == pre) {
          const uint32_t at = atomicAdd(&sm.count, 1u);
          sm.ckey[at] = kr[j];
          sm.cidx[at] = base + 32 * j;
        }
      }
    }
    const uint32_t need = sm.need;
    __syncthreads();
    for (int c = tid; c < cand; c += NT) {  // the token of rank need - 1 in the bin
      const uint32_t x = sm.ckey[c];
      const int32_t i = sm.cidx[c];
      uint32_t more = 0, same = 0;  // keys above this one, equal ones before it
      for (int e = 0; e < cand; e += 4) {
        const uint4 y = *(const uint4*)&sm.ckey[e];
        const int4 p = *(const int4*)&sm.cidx[e];
        more += (y.x > x) + (y.y > x) + (y.z > x) + (y.w > x);
        same += (y.x == x && p.x < i) + (y.y == x && p.y < i) + (y.z == x && p.z < i) + (y.w == x && p.w < i);
      }
      if (more + same == need - 1) {
        sm.T = x;
        sm.need = same + 1;
      }
    }
    __syncthreads();
    T = sm.T;
  }
  TRC_ADD(1, tr_r);
  TRC_T(tr_e);
  // ---- emission, slab by slab ----
  const uint32_t nties = sm.need;
  uint32_t run = 0, eq_run = 0;  // keys > T and == T before this slab
#pragma unroll 1
  for (int sl = 0; sl < nslab; ++sl) {
    if (nslab > 1) load_slab<KPT, NT>(key, n, sl, warp, lane, kr);
    const int first = sl * SLAB + warp * (32 * KPT);
    // the tokens > T and == T of slot `lane` (keys past the request's end are 0 in kr:
    // not above T, and the last of any ties)
    uint32_t mine = 0, eq = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const uint32_t b = __ballot_sync(0xffffffffu, kr[j] > T);
      const uint32_t e = __ballot_sync(0xffffffffu, kr[j] == T);
      if (lane == j) {
        mine = b;
        eq = e;
      }
    }
    // prefixes over lanes, then warps: keys > T in the low half, ties in the high one
    // (a slab has at most 32768 keys)
    const uint32_t c = __popc(mine) | (uint32_t)__popc(eq) << 16;
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    uint32_t* tot = sm.tot[sl & 1];
    if (lane == 31) tot[warp] = inc;
    __syncthreads();
    const uint32_t w = lane < NW ? tot[lane] : 0u;
    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + inc - c;
    const uint32_t all = __reduce_add_sync(0xffffffffu, w);
    const uint32_t eb = eq_run + (before >> 16);  // ties before the lane's
    uint32_t at = run + (before & 0xffffu) + min(eb, nties);
    run += all & 0xffffu;
    eq_run += all >> 16;
    for (uint32_t take = eb < nties ? min(nties - eb, (uint32_t)__popc(eq)) : 0u; take != 0; --take) {
      mine |= eq & (0u - eq);
      eq &= eq - 1;
    }
    while (mine != 0) {
      const int i = first + 32 * lane + __ffs(mine) - 1;
      mine &= mine - 1;
      if (at < (uint32_t)B) {
        out[at] = i;
        if (at < SE_IDX) sm.idx[at] = i;
      }
      ++at;
    }
  }
  __syncthreads();  // the positions are read back below
  TRC_ADD(2, tr_e);
  TRC_T(tr_g);
  if constexpr (GATHER) gather_unit<E, NT>(dm, plane, start, end, true, k, v, out, sm.idx, B, u, part, parts, k_out,
                                          v_out);
  TRC_ADD(3, tr_g);
  if constexpr (MODE == 2) {
    // f = the kept positions below B (they ascend: a binary search)
    int lo = 0, hi = B;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((mid < SE_IDX ? sm.idx[mid] : out[mid]) < B) lo = mid + 1; else hi = mid;
    }
    fill_holes_unit<E, NT>(dm, plane, start, B, lo, part, parts, kio, vio, pos, out);
  }
  TRC_ADD(5, tr_u);
  if (tid == 0) TRC_PUT(ws, TR_K_SELECT, 6);
}

template <typename T>
__global__ void __launch_bounds__(256)
    compact_kernel(Dims dm, const int32_t* __restrict__ cu, const T* __restrict__ k, const T* __restrict__ v,
                   const int32_t* __restrict__ idx, int B, T* __restrict__ k_out, T* __restrict__ v_out) {
  pdl_wait();
  constexpr int CH = D * (int)sizeof(T) / 16;  // 16-byte chunks per row
  const int64_t rows = (int64_t)dm.L * dm.Hkv * dm.S * B;
  const int64_t total = rows * CH;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / CH;
    const int c = (int)(e % CH);
    const int64_t u = row / B;
    const int plane = (int)(u / dm.S), s = (int)(u % dm.S);
    const int l = plane / dm.Hkv, g = plane % dm.Hkv;
    const int32_t src = idx[row];
    const int64_t start = cu[s], end = cu[s + 1];
    uint4 kk = make_uint4(0, 0, 0, 0), vv = make_uint4(0, 0, 0, 0);
    // positions outside the request (or a malformed cu_seqlens) give zero rows
    if (src >= 0 && start >= 0 && start + src < end && end <= dm.Ntot) {
      const int64_t off = (int64_t)l * dm.kv_sl + (int64_t)g * dm.kv_sh + ((int64_t)cu[s] + src) * dm.kv_st;
      kk = *((const uint4*)(k + off) + c);
      vv = *((const uint4*)(v + off) + c);
    }
    *((uint4*)(k_out + row * D) + c) = kk;
    *((uint4*)(v_out + row * D) + c) = vv;
  }
}

template <int KPT, int NT>
static cudaError_t launch_select_kpt(const Dims& dm, const Ws& ws, const int32_t* cu, const float* scores, int budget,
                                     int32_t* idx, int32_t* kept, int dtype, const void* k, const void* v,
                                     void* k_out, void* v_out, void* kio, void* vio, int32_t* pos, int grid, int parts,
                                     cudaStream_t st) {
  using bf = __nv_bfloat16;
  if (kio != nullptr) {  // hole filling in place
    if (dtype == 1)
      return launch_pdl(dm.pdl != 0, select_kernel<KPT, bf, 2, NT>, grid, NT, 0, st, dm, ws, cu, scores, budget,
                        idx, kept, (const bf*)nullptr, (const bf*)nullptr, (bf*)nullptr, (bf*)nullptr, (bf*)kio,
                        (bf*)vio, pos, parts);
    return launch_pdl(dm.pdl != 0, select_kernel<KPT, float, 2, NT>, grid, NT, 0, st, dm, ws, cu, scores, budget,
                      idx, kept, (const float*)nullptr, (const float*)nullptr, (float*)nullptr, (float*)nullptr,
                      (float*)kio, (float*)vio, pos, parts);
  }
  if (k == nullptr)
    return launch_pdl(dm.pdl != 0, select_kernel<KPT, bf, 0, NT>, grid, NT, 0, st, dm, ws, cu, scores, budget,
                      idx, kept, (const bf*)nullptr, (const bf*)nullptr, (bf*)nullptr, (bf*)nullptr, (bf*)nullptr,
                      (bf*)nullptr, (int32_t*)nullptr, parts);
  if (dtype == 1)
    return launch_pdl(dm.pdl != 0, select_kernel<KPT, bf, 1, NT>, grid, NT, 0, st, dm, ws, cu, scores, budget,
                      idx, kept, (const bf*)k, (const bf*)v, (bf*)k_out, (bf*)v_out, (bf*)nullptr, (bf*)nullptr,
                      (int32_t*)nullptr, parts);
  return launch_pdl(dm.pdl != 0, select_kernel<KPT, float, 1, NT>, grid, NT, 0, st, dm, ws, cu, scores, budget,
                    idx, kept, (const float*)k, (const float*)v, (float*)k_out, (float*)v_out, (float*)nullptr,
                    (float*)nullptr, (int32_t*)nullptr, parts);
}

cudaError_t launch_select(const Dims& dm, const Ws& ws, const int32_t* cu, const float* scores, int budget,
                          int32_t* idx, int32_t* kept, int max_seqlen, cudaStream_t st, int dtype,
                          const void* k, const void* v, void* k_out, void* v_out, void* kio, void* vio,
                          int32_t* pos) {
#define JACAP_SELECT(KPT, NT)                                                                                   \
  JACAP_TRY((launch_select_kpt<KPT, NT>(dm, ws, cu, scores, budget, idx, kept, dtype, k, v, k_out, v_out, kio, vio, \
                                        pos, grid, parts, st)))
  // More units than SMs: CTAs of 256 threads (four per SM) while they hold the
  // longest request in one slab, of 512 (two per SM) beyond that (256 units of 32768
  // tokens: 42 us, 46 with 1024 threads; of 131072: 119 and 120). Otherwise CTAs of
  // 1024 threads, as many per unit as there are SMs for (112 units of 20011 tokens,
  // 2048 kept: 51 us; 60 with two CTAs of 512 threads each).
  int dev = 0, sms = 0;
  JACAP_TRY(cudaGetDevice(&dev));
  JACAP_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t units = (int64_t)dm.L * dm.Hkv * dm.S;
  if (units >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
  const bool many = units > sms;
  const int parts = many || (k == nullptr && kio == nullptr)
                        ? 1
                        : (int)std::max<int64_t>(1, std::min<int64_t>(sms / units, budget / 32));
  const int grid = (int)units * parts;
  if (many && max_seqlen <= 256 * 4) JACAP_SELECT(4, 256);
  else if (many && max_seqlen <= 256 * 8) JACAP_SELECT(8, 256);
  else if (many && max_seqlen <= 256 * 16) JACAP_SELECT(16, 256);
  else if (many && max_seqlen <= 256 * 32) JACAP_SELECT(32, 256);
  else if (many) JACAP_SELECT(32, 512);
  else if (max_seqlen <= 1024 * 4) JACAP_SELECT(4, 1024);
  else if (max_seqlen <= 1024 * 8) JACAP_SELECT(8, 1024);
  else if (max_seqlen <= 1024 * 16) JACAP_SELECT(16, 1024);
  else JACAP_SELECT(32, 1024);
#undef JACAP_SELECT
  return cudaGetLastError();
}

cudaError_t launch_compact(const Dims& dm, int dtype, const int32_t* cu, const void* k, const void* v,
                           const int32_t* idx, int budget, void* k_out, void* v_out, cudaStream_t st) {
  const int64_t rows = (int64_t)dm.L * dm.Hkv * dm.S * budget;
  const int es = dtype == 1 ? 2 : 4;
  const int64_t total = rows * (D * es / 16);
  const int64_t blocks64 = (total + 255) / 256;
  const int blocks = (int)(blocks64 < 65535 * 16 ? blocks64 : 65535 * 16);
  if (blocks <= 0) return cudaSuccess;
  if (dtype == 1)
    JACAP_TRY(launch_pdl(dm.pdl != 0, compact_kernel<__nv_bfloat16>, blocks, 256, 0, st, dm, cu,
                         (const __nv_bfloat16*)k, (const __nv_bfloat16*)v, idx, budget, (__nv_bfloat16*)k_out,
                         (__nv_bfloat16*)v_out));
  else
    JACAP_TRY(launch_pdl(dm.pdl != 0, compact_kernel<float>, blocks, 256, 0, st, dm, cu, (const float*)k,
                         (const float*)v, idx, budget, (float*)k_out, (float*)v_out));
  return cudaGetLastError();
}

}  // namespace jacap
