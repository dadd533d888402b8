// k_score.cu - Jacap scores r_i = w_i v_i^T A^{-1} v_i = w_i ||L^{-1} v_i||^2 (Eq. 10).
//
// bf16 caches: the tensor cores form Y = V (L^{-1})^T for a 128-token tile
// from hi(L^{-1}) and lo(L^{-1}) (K-major, from a 64 KB shared-memory image
// written by the factor kernel, hi and lo interleaved by 16-row blocks).
// L^{-1} is lower triangular, so output row n needs only channels <= n: the
// K-step of channels 16 k .. 16 k + 15 is one MMA of N = 256 - 32 k over the
// image rows (hi and lo of output rows 16 k .. 127) into accumulator columns
// 32 k .. 255, eight MMAs per tile in all. The image's rows 0-127 of channels
// 64-127 (output rows 0-63) are zero and not copied into shared memory, which
// leaves room for a fourth V stage. V comes straight from the TMA-staged tile;
// a warp of its own loads the images, so the V ring never waits behind an
// image slot. Each epilogue thread owns one token (one TMEM lane) and reduces
// ||y||^2 = sum_n (hi_n + lo_n)^2 in fp32, then multiplies by w_i. (With
// output directions the matrix is full: hi and lo accumulate into the same
// 128 columns, four MMAs of N = 128 per K-step pair.) The tensor-memory accumulator
// is double-buffered so the epilogue of tile i overlaps the MMAs of tile i+1,
// and so is the L^{-1} image: it is loaded once per run of consecutive items
// of one unit, and the next unit's image streams in while the current run's
// tiles go through.
// float32 caches: SIMT forward products with L^{-1} held in shared memory.
#include "jacap_dev.cuh"
#include "jacap_internal.h"
#include "k_score_body.cuh"

namespace jacap {

template <bool DENSE>
__global__ void __launch_bounds__(SC_THREADS, 1)
    score_bf16_kernel(const __grid_constant__ CUtensorMap vmap, Dims dm, Ws ws, const int32_t* __restrict__ cu,
                      float* __restrict__ scores) {
  pdl_wait();
  score_bf16_body<DENSE, false>(&vmap, dm, ws, scores, blockIdx.x, gridDim.x);
}

// ------------------------------------------------------------ SIMT fp32 ---
// Y = V (L^{-1})^T for a 128-token tile: a warp takes the output rows 8 w .. + 7 and
// 8 (15 - w) .. + 7 (together 136 columns of the triangle for every warp), a lane
// the tokens lane + 32 j, so that each 16-byte read of L^{-1} (one address for the
// warp) serves 16 multiply-adds and each of V 32. L^{-1} is stored with zeros above
// the diagonal, so a block of 8 rows may run its columns up to its last row. The
// warps' partial sums of squares meet in shared memory, added in warp order. The
// next tile's V streams in (16-byte asynchronous copies) while this one is worked on.
// Bound: the issue of float32 multiply-adds, 4352 per warp and tile, 8704 cycles per
// tile and sub-partition (two warps). 8 x 4096 tokens: 0.055 -> 0.025 ms against two
// threads per token with four rows each.
constexpr int SF_THREADS = 256;
constexpr int SF_LD = D + 4;
constexpr size_t score_f32_smem_bytes() { return ((size_t)D * D + 2 * TILE * SF_LD + 8 * TILE) * sizeof(float); }

__global__ void __launch_bounds__(SF_THREADS, 1)
    score_f32_kernel(Dims dm, Ws ws, const int32_t* __restrict__ cu, const float* __restrict__ v,
                     float* __restrict__ scores) {
  pdl_wait();
  extern __shared__ __align__(16) float ssm[];
  float* Mi = ssm;                       // [D][D] L^{-1}
  float* vt = ssm + D * D;               // [2][TILE][SF_LD]
  float* red = vt + 2 * TILE * SF_LD;    // [8 warps][TILE]
  __shared__ int s_skip;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) s_skip = status_failed(ws) ? 1 : 0;
  __syncthreads();
  if (s_skip) return;
  bool bad = false;
  // the CTA's tiles, one ahead: (item, t) is the tile being worked on, (nitem, nt) the next
  ItemStream is(dm, ws, blockIdx.x, gridDim.x);
  Item item, nitem;
  bool more = is.next(nitem);
  int64_t t = 0, nt = more ? nitem.t0 : 0;
  auto fetch = [&](int buf) {  // the next tile's V into buffer `buf`
    const int l = nitem.plane / dm.Hkv, g = nitem.plane % dm.Hkv;
    const float* src = v + (int64_t)l * dm.kv_sl + (int64_t)g * dm.kv_sh + nt * dm.kv_st;
    const int nv = (int)(nitem.t1 - nt < TILE ? nitem.t1 - nt : TILE);
    float* dst = vt + buf * TILE * SF_LD;
#pragma unroll 4
    for (int e = tid; e < TILE * (D / 4); e += SF_THREADS) {
      const int r = e / (D / 4), c4 = (e % (D / 4)) * 4;
      cp_async16(smem_u32(dst + r * SF_LD + c4), src + (r < nv ? r : 0) * dm.kv_st + c4, r < nv);
    }
  };
  if (more) fetch(0);
  cp_async_commit();
  int64_t loaded = -1;
  for (int buf = 0; more; buf ^= 1) {
    item = nitem;
    t = nt;
    const int64_t u = (int64_t)item.plane * dm.S + item.seq;
    if (u != loaded) {  // the previous tile's reads of L^{-1} ended at its last barrier
      const float* src = ws.minv + u * D * D;
#pragma unroll 4
      for (int e = tid * 4; e < D * D; e += SF_THREADS * 4) cp_async16(smem_u32(Mi + e), src + e, true);
      loaded = u;
    }
    cp_async_commit();
    nt += TILE;
    if (nt >= item.t1) {
      more = is.next(nitem);
      if (more) nt = nitem.t0;
    }
    if (more) fetch(buf ^ 1);
    cp_async_commit();
    cp_async_wait<1>();  // this tile and L^{-1} are here
    __syncthreads();
    const float* vb = vt + buf * TILE * SF_LD + lane * SF_LD;
    float ssq[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const int blk = half == 0 ? warp : 15 - warp;
      const float* m0 = Mi + 8 * blk * D;
      const int cend = dm.dense_minv ? D : 8 * blk + 8;  // a full matrix with output directions
      float y[4][8];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int r = 0; r < 8; ++r) y[j][r] = 0.f;
#pragma unroll 1
      for (int c = 0; c < cend; c += 4) {
        float4 x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = *(const float4*)(vb + 32 * j * SF_LD + c);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const float4 a = *(const float4*)(m0 + r * D + c);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            y[j][r] = fmaf(a.w, x[j].w, fmaf(a.z, x[j].z, fmaf(a.y, x[j].y, fmaf(a.x, x[j].x, y[j][r]))));
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int r = 0; r < 8; ++r) ssq[j] = fmaf(y[j][r], y[j][r], ssq[j]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) red[warp * TILE + lane + 32 * j] = ssq[j];
    __syncthreads();
    if (tid < TILE && t + tid < item.t1) {
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < 8; ++w) sum += red[w * TILE + tid];
      const int64_t o = (int64_t)item.plane * dm.Ntot + t + tid;
      const float sc = ws.w[o] * sum;
      scores[o] = sc;
      bad |= !isfinite(sc);
    }
    __syncthreads();  // red and this tile's buffer are free
  }
  cp_async_wait<0>();
  if (bad) flag(ws, ST_NONFINITE);
}

cudaError_t launch_score(const CUtensorMap& vmap, const Dims& dm, const Ws& ws, int dtype, const void* v,
                         const int32_t* cu, float* scores, int grid, cudaStream_t st) {
  if (dtype == 1) {
    const size_t smem = dm.dense_minv ? score_bf16_smem_bytes<true>() : score_bf16_smem_bytes<false>();
    static_assert(score_bf16_smem_bytes<true>() + 512 <= 232448 && score_bf16_smem_bytes<false>() + 512 <= 232448,
                  "shared memory");  // 512: the static variables
    auto kern = dm.dense_minv ? score_bf16_kernel<true> : score_bf16_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    JACAP_TRY(launch_pdl(dm.pdl != 0, kern, grid, SC_THREADS, smem, st, vmap, dm, ws, cu, scores));
  } else {
    constexpr size_t smem = score_f32_smem_bytes();
    cudaError_t e = cudaFuncSetAttribute(score_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    JACAP_TRY(launch_pdl(dm.pdl != 0, score_f32_kernel, grid, SF_THREADS, smem, st, dm, ws, cu, (const float*)v,
                         scores));
  }
  return cudaGetLastError();
}

}  // namespace jacap
