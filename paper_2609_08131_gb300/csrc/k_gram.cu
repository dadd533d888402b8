// k_gram.cu - Jacobian weights and the weighted Gram pass over V.
//
// Weight pass (float32 caches; one streaming pass over the K pass's logits/kappa
// rows; with bf16 caches the Gram kernel forms the same weights itself), per work
// item (a chunk of one unit's tokens):
//   1. combines the K pass's per-chunk (max, sum exp) into the pool-softmax
//      normaliser (M_h, Z_h) of each query head h of the group (Sec. 3.4,
//      display after Algorithm 1);
//   2. forms w_i = (1/d) sum_h [alpha_bar (1 - alpha_bar)]^2 kappa_h,i with
//      alpha_bar = exp(l_h,i - M_h) / Z_h (Eq. 8; GQA heads summed) and stores
//      w for the score pass and as a bf16 pair hi + lo for the Gram pass.
// Gram pass: accumulates a partial Gram per run of chunks,  sum_i w_i v_i v_i^T  (Eq. 9).
//
// bf16 caches use the 5th-generation tensor cores. B = V straight from the
// TMA-staged tile (bf16 is exact); the scaled operand w_i v_i = hi + lo is
// split into two bf16 halves (residual ~2^-17 relative per product) by the
// scaling warps with packed bf16 arithmetic on w_i = whi + wlo, and written to
// tensor memory as two A operands, so
// D = sum_i (hi_i + lo_i) v_i^T accumulates in fp32 in tensor memory without
// passing the scaled operand through shared memory. float32 caches take a
// SIMT fp32 kernel of the same contract.
#include "jacap_dev.cuh"
#include "jacap_internal.h"
#include "k_gram_body.cuh"

namespace jacap {

// ---------------------------------------------------------------- weights --
// w_i of Eq. 8 summed over the G query heads of the group (GQA heads add their
// weights): w_i = wdiv * sum_h [alpha_bar (1 - alpha_bar)]^2 kappa_h,i with
// alpha_bar = exp(l_h,i - M_h) / Z_h; with the linear surrogate (S_C = I)
// rho = 1 and w_i = wdiv * sum_h kappa_h,i. One streaming pass over the K pass's
// logits/kappa rows that writes w, for float32 caches (with bf16 caches the
// tensor-core Gram computes the same weights itself).
constexpr int WT_THREADS = 256;

template <int G>
__global__ void __launch_bounds__(WT_THREADS) weight_kernel(Dims dm, Ws ws, const int32_t* __restrict__ cu) {
  pdl_wait();
  __shared__ int s_skip;
  const int tid = threadIdx.x;
  if (tid == 0) s_skip = status_failed(ws) ? 1 : 0;
  __syncthreads();
  if (s_skip) return;
  bool bad = false, cont = false;
  float u[2 * G];
  Item item;
  for (ItemStream is(dm, ws, blockIdx.x, gridDim.x); is.next(item);) {
    if (!cont) load_unit_stats<G>(dm, ws, item.plane, item.seq, u);  // a new unit: its (M_h, 1 / Z_h)
    cont = is.next_same_unit(item);
    const int64_t base = (int64_t)item.plane * dm.Ntot;
    // four tokens per thread per round, their loads issued together
    for (int64_t t4 = item.t0 + tid; t4 < item.t1; t4 += 4 * WT_THREADS) {
      float lk[4][2 * G];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t tok = t4 + q * WT_THREADS;
        const float* src = ws.lk + (base + (tok < item.t1 ? tok : t4)) * (2 * G);
        load_floats<2 * G, LkAlign<G>::ROW>(lk[q], src);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t tok = t4 + q * WT_THREADS;
        if (tok >= item.t1) break;
        float wt = 0.f;
        if (dm.linear) {  // S_C = I: rho = 1
#pragma unroll
          for (int h = 0; h < G; ++h) wt += lk[q][G + h];
        } else {
#pragma unroll
          for (int h = 0; h < G; ++h) {
            const float a = expf(lk[q][h] - u[h]) * u[G + h];  // alpha_bar
            const float rho = a * (1.f - a);                    // diagonal of the softmax Jacobian
            wt = fmaf(rho * rho, lk[q][G + h], wt);             // rho^2 kappa
          }
        }
        wt *= dm.wdiv;
        bad |= !isfinite(wt);
        ws.w[base + tok] = wt;
      }
    }
  }
  if (bad) flag(ws, ST_NONFINITE);
}

template <int G>
__global__ void __launch_bounds__(GR_THREADS, 1)
    gram_bf16_kernel(const __grid_constant__ CUtensorMap vmap, Dims dm, Ws ws, const int32_t* __restrict__ cu) {
  pdl_wait();
  gram_bf16_body<G, false>(&vmap, dm, ws, blockIdx.x, gridDim.x);
}

// ------------------------------------------------------------ SIMT fp32 ---
// float32 caches: a thread accumulates one 8 x 4 tile that reaches the Gram's
// diagonal or lies below it (272 tiles, rows 8 ty .., columns 4 cx ..; nine warps
// spread evenly over the sub-partitions) over 128-token tiles of V in
// shared memory, fetched with 16-byte asynchronous copies (three CTAs per SM cover
// each other's fetches). Bound: float32 multiply-adds, 32 per token and thread
// beside three 16-byte shared-memory reads. 8 x 4096 tokens: 0.039 -> 0.025 ms
// against all 256 tiles over slabs of 32 tokens staged through registers.
constexpr int GF_THREADS = 288;
constexpr int GF_TILES = 272;
constexpr int GF_LD = D + 4;
constexpr size_t GF_SMEM = ((size_t)TILE * GF_LD + TILE) * sizeof(float);

__global__ void __launch_bounds__(GF_THREADS, 3)
    gram_f32_kernel(Dims dm, Ws ws, const int32_t* __restrict__ cu, const float* __restrict__ v) {
  pdl_wait();
  extern __shared__ __align__(16) float gsm[];
  float* vs = gsm;                 // [TILE][GF_LD]
  float* wsl = gsm + TILE * GF_LD;  // [TILE]
  __shared__ int s_skip;
  const int tid = threadIdx.x;
  if (tid == 0) s_skip = status_failed(ws) ? 1 : 0;
  __syncthreads();
  if (s_skip) return;
  // tiles 0 .. ty (ty + 1) - 1 lie in the tile rows above ty
  int ty = (int)((sqrtf(4.f * (float)tid + 1.f) - 1.f) * 0.5f);
  while (ty * (ty + 1) > tid) --ty;
  while ((ty + 1) * (ty + 2) <= tid) ++ty;
  const int cx = tid - ty * (ty + 1);
  const bool own = tid < GF_TILES;
  Item item;
  for (ItemStream is(dm, ws, blockIdx.x, gridDim.x); is.next(item);) {
    const int l = item.plane / dm.Hkv, g = item.plane % dm.Hkv;
    const float* vbase = v + (int64_t)l * dm.kv_sl + (int64_t)g * dm.kv_sh;
    float2 acc[8][2];  // columns (2 q, 2 q + 1) of row p
#pragma unroll
    for (int p = 0; p < 8; ++p) acc[p][0] = acc[p][1] = make_float2(0.f, 0.f);
    for (int64_t t = item.t0; t < item.t1; t += TILE) {
      const int nv = (int)(item.t1 - t < TILE ? item.t1 - t : TILE);
      for (int e = tid; e < TILE * (D / 4); e += GF_THREADS) {
        const int r = e / (D / 4), c4 = (e % (D / 4)) * 4;
        cp_async16(smem_u32(vs + r * GF_LD + c4), vbase + (t + (r < nv ? r : 0)) * dm.kv_st + c4, r < nv);
      }
      if (tid < TILE) wsl[tid] = tid < nv ? ws.w[(int64_t)item.plane * dm.Ntot + t + tid] : 0.f;
      cp_async_commit();
      cp_async_wait<0>();
      __syncthreads();
      if (own) {
#pragma unroll 2
        for (int r = 0; r < nv; ++r) {
          const float wt = wsl[r];
          const float4 a0 = *(const float4*)(vs + r * GF_LD + 8 * ty), a1 = *(const float4*)(vs + r * GF_LD + 8 * ty + 4);
          const float4 b = *(const float4*)(vs + r * GF_LD + 4 * cx);
          const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
          const float2 x[2] = {make_float2(wt * b.x, wt * b.y), make_float2(wt * b.z, wt * b.w)};  // w v of the columns
#pragma unroll
          for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int q = 0; q < 2; ++q) acc[p][q] = __ffma2_rn(make_float2(a[p], a[p]), x[q], acc[p][q]);
        }
      }
      __syncthreads();  // the tile is read before the next one lands on it
    }
    float* dst = ws.gpart + ((int64_t)item.plane * dm.c_cap + item.cidx) * D * D;
    if (tid == 0) ws.pflag[(int64_t)item.plane * dm.c_cap + item.cidx] = 1;  // a partial per chunk here
    if (own) {
#pragma unroll
      for (int p = 0; p < 8; ++p) {
        // (m, n) at ((n / 32) D + m) 32 + n % 32
        *(float4*)(dst + ((cx >> 3) * D + 8 * ty + p) * 32 + (cx & 7) * 4) =
            make_float4(acc[p][0].x, acc[p][0].y, acc[p][1].x, acc[p][1].y);
      }
    }
  }
}

// ------------------------------------------------------- unit statistics --
// Warp h of block u merges the chunk statistics of unit u for query head h
// (unit_softmax_stats_warp) and stores (M_h, 1 / Z_h) in ws.ustats, so the
// weight computations read two floats per head instead of merging the unit's
// chunks themselves at every unit they start.
template <int G>
__global__ void __launch_bounds__(32 * G) unit_stats_kernel(Dims dm, Ws ws) {
  pdl_wait();
  if (status_failed(ws)) return;
  const int u = blockIdx.x, h = threadIdx.x >> 5;
  float M, Z;
  unit_softmax_stats_warp<G>(dm, ws, u / dm.S, u % dm.S, h, M, Z);
  if ((threadIdx.x & 31) == 0) {
    ws.ustats[(int64_t)u * 2 * G + h] = M;
    ws.ustats[(int64_t)u * 2 * G + G + h] = 1.f / Z;
  }
}

template <int G>
static cudaError_t launch_unit_stats_g(const Dims& dm, const Ws& ws, cudaStream_t st) {
  JACAP_TRY(launch_pdl(dm.pdl != 0, unit_stats_kernel<G>, dm.L * dm.Hkv * dm.S, 32 * G, 0, st, dm, ws));
  return cudaGetLastError();
}

cudaError_t launch_unit_stats(const Dims& dm, const Ws& ws, cudaStream_t st) {
  switch (dm.G) {
    case 1: return launch_unit_stats_g<1>(dm, ws, st);
    case 2: return launch_unit_stats_g<2>(dm, ws, st);
    case 3: return launch_unit_stats_g<3>(dm, ws, st);
    case 4: return launch_unit_stats_g<4>(dm, ws, st);
    case 5: return launch_unit_stats_g<5>(dm, ws, st);
    case 6: return launch_unit_stats_g<6>(dm, ws, st);
    case 7: return launch_unit_stats_g<7>(dm, ws, st);
    case 8: return launch_unit_stats_g<8>(dm, ws, st);
    default: return cudaErrorInvalidValue;
  }
}

// ------------------------------------------------------------ launchers ----
template <int G>
static cudaError_t launch_weights_g(const Dims& dm, const Ws& ws, const int32_t* cu, int grid, cudaStream_t st) {
  JACAP_TRY(launch_pdl(dm.pdl != 0, weight_kernel<G>, grid, WT_THREADS, 0, st, dm, ws, cu));
  return cudaGetLastError();
}

cudaError_t launch_weights(const Dims& dm, const Ws& ws, const int32_t* cu, int grid, cudaStream_t st) {
  switch (dm.G) {
    case 1: return launch_weights_g<1>(dm, ws, cu, grid, st);
    case 2: return launch_weights_g<2>(dm, ws, cu, grid, st);
    case 3: return launch_weights_g<3>(dm, ws, cu, grid, st);
    case 4: return launch_weights_g<4>(dm, ws, cu, grid, st);
    case 5: return launch_weights_g<5>(dm, ws, cu, grid, st);
    case 6: return launch_weights_g<6>(dm, ws, cu, grid, st);
    case 7: return launch_weights_g<7>(dm, ws, cu, grid, st);
    case 8: return launch_weights_g<8>(dm, ws, cu, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int G>
static cudaError_t launch_gram_bf16(const CUtensorMap& vmap, const Dims& dm, const Ws& ws, const int32_t* cu,
                                   int grid, cudaStream_t st) {
  constexpr size_t smem = GrCfg<G>::SMEM;
  cudaError_t e = cudaFuncSetAttribute(gram_bf16_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  JACAP_TRY(launch_pdl(dm.pdl != 0, gram_bf16_kernel<G>, grid, GR_THREADS, smem, st, vmap, dm, ws, cu));
  return cudaGetLastError();
}

cudaError_t launch_gram(const CUtensorMap& vmap, const Dims& dm, const Ws& ws, int dtype, const void* v,
                        const int32_t* cu, int grid, cudaStream_t st) {
  if (dtype == 1) {
    switch (dm.G) {
      case 1: return launch_gram_bf16<1>(vmap, dm, ws, cu, grid, st);
      case 2: return launch_gram_bf16<2>(vmap, dm, ws, cu, grid, st);
      case 3: return launch_gram_bf16<3>(vmap, dm, ws, cu, grid, st);
      case 4: return launch_gram_bf16<4>(vmap, dm, ws, cu, grid, st);
      case 5: return launch_gram_bf16<5>(vmap, dm, ws, cu, grid, st);
      case 6: return launch_gram_bf16<6>(vmap, dm, ws, cu, grid, st);
      case 7: return launch_gram_bf16<7>(vmap, dm, ws, cu, grid, st);
      case 8: return launch_gram_bf16<8>(vmap, dm, ws, cu, grid, st);
      default: return cudaErrorInvalidValue;
    }
  } else {
    JACAP_TRY(cudaFuncSetAttribute(gram_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GF_SMEM));
    JACAP_TRY(launch_pdl(dm.pdl != 0, gram_f32_kernel, grid, GF_THREADS, GF_SMEM, st, dm, ws, cu, (const float*)v));
  }
  return cudaGetLastError();
}

}  // namespace jacap
