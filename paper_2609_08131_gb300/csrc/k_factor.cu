// k_factor.cu - capacity matrix and the inverse of its Cholesky factor, one
// CTA per unit.
//
//  G        = sum over the unit's chunks of the partial Grams  (Eq. 9 without I)
//  A        = I + G                                           (Eq. 9, Sigma_noise = I)
//  L^{-1}   where A = L L^T.
//
// Since v^T A^{-1} v = ||L^{-1} v||^2, the score pass needs only L^{-1}
// (Eq. 10). It is obtained by block forward elimination of [A | I] without
// pivoting (safe: A is symmetric positive definite), four rows at a time, in
// place in registers: a thread holds the tile of rows 8 ty .. + 7 and columns
// 4 cx .. + 3 of one 128 x 128 array, whose column c holds A until its block is
// eliminated and the inverse's part afterwards; the 272 tiles that reach the
// diagonal or lie below it are dealt to 9 warps row by row, so that few lanes
// idle and whole warps leave as the elimination goes down. Step b (block rows and
// columns 4 b .. 4 b + 3, Cholesky factor L_b of the pivot block):
//   u_c = L_b^{-1} A_cb^T  (c below the block)
//   u_c = L_b^{-1} Z_bc    (c before it): the final rows of L^{-1}
//   u_c = column of L_b^{-1} (c in it)
//   Z_rc -= u_r . u_c      for every row r below the block and c <= r (from 0 in the block's columns)
// The array holds A - I, and each pivot block gets its I when its turn comes: where
// G is small beside I (long caches), the updates round at G's size and not at 1's.
// The tiles that own the vectors leave them in shared memory when they have made
// their update of the step before, the pivot's owner L_b^{-1}; threads 0-127 turn
// one vector each into u (two barriers a step), and every tile below makes the
// same rank-4 update.
//
// Bound: the chain of the 32 steps, 1240 cycles each alone on an SM (barriers 170,
// vectors left and turned into u 500, the pivot block's four reciprocals 170, the
// update 400) and 760 (650, 610) per unit with two (three, four) CTAs on an SM;
// with many units also the 192 KB that each writes. Measured against blocked 32 x 32
// eliminations of one warp each, with the blocks in shared memory: 256 units 0.055 ->
// 0.042 ms, 448 units 0.082 -> 0.060, 1024 units 0.173 -> 0.120; output directions,
// 128 units, 0.124 -> 0.070 ms. 8 x 8 tiles whose owners formed u themselves took
// 0.061 and 0.192 ms (two lanes a warp formed eight vectors each); tiles paired by
// columns, whose rows' values all had to be doubled, 1360 cycles a step.
//
// With output directions u = W v (Sec. 3.1) the capacity matrix I + sum w u u^T
// lives in the output space; with a 128 x 128 factor F of W^T W (F^T F = W^T W)
// it reduces exactly to M = I + F G F^T, and u^T A^{-1} u = ||L_M^{-1} F v||^2.
// That variant (PROJ) forms F G with 8 x 8 register tiles (operands in shared
// memory) and the tiles that the elimination holds of F (F G)^T straight in their
// owners' registers, factors M as above and writes T = L_M^{-1} F, a third product
// (to the diagonal only), in place of L^{-1}. Full 128 x 128 x 128 for the last two,
// M by way of shared memory: 0.080 ms for 128 units instead of 0.070.
//
// L^{-1} is written twice: as float32 (used by the float32 score pass and
// exposed for tests) and as a bf16 hi/lo pair laid out exactly as the
// shared-memory B operand of the tensor-core score pass (K-major, 128-byte
// swizzle, two 64-channel atoms of 256 rows): hi(L^{-1}[n, :]) at row
// 32 (n / 16) + n % 16 and lo(L^{-1}[n, :]) = L^{-1} - hi rounded again 16
// rows further (hi and lo interleaved by 16-row blocks, so the rows a K-step
// of the triangular product needs are contiguous), so hi + lo carries ~16
// significant bits. The output-direction variant (T = L_M^{-1} F, a full
// matrix) keeps hi in rows 0-127 and lo in rows 128-255. Both go straight from the
// tiles' registers.
#include "jacap_dev.cuh"
#include "jacap_internal.h"

namespace jacap {

constexpr int FT_TILES = 272;     // tiles (ty, cx), cx <= 2 ty + 1
constexpr int FT_THREADS = 288;
constexpr int FT_TRACED = 240;    // (time accounting) the owner of the last tile row's first tile: in every step

// A step's vectors: raw by index (16 bytes between the tile rows, so that the rows
// that a warp stores fall in different banks), u by component.
struct FtSmem {
  float4 raw[D + D / 8];
  float4 linv[4];
  float ut[4][D];
  int list[FT_THREADS];
  int cnt[FT_THREADS / 32];
  int skip;
};

// 4 pairs of rows, 4 columns: the packed multiply-adds of a rank-1 update then take
// the rows' vector in pairs as it is loaded, and only the columns' 4 values doubled.
using Tile = float2[4][4];

__device__ __forceinline__ float& tile_at(Tile& T, int i, int c) {  // i, c known after unrolling
  return (i & 1) ? T[i >> 1][c].y : T[i >> 1][c].x;
}
__device__ __forceinline__ float4 tile_row(Tile& T, int i) {
  return make_float4(tile_at(T, i, 0), tile_at(T, i, 1), tile_at(T, i, 2), tile_at(T, i, 3));
}
__device__ __forceinline__ void tile_set_row(Tile& T, int i, const float4 v) {
  tile_at(T, i, 0) = v.x, tile_at(T, i, 1) = v.y, tile_at(T, i, 2) = v.z, tile_at(T, i, 3) = v.w;
}

// 1 / sqrt(x): the hardware's approximation refined by one Newton-Raphson step;
// 1 / x likewise.
__device__ __forceinline__ float rsqrt_nr(float x) {
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);
}
__device__ __forceinline__ float rcp_nr(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return fmaf(y, fmaf(-x, y, 1.f), y);
}

// L_b^{-1} of the pivot block in rows O .. O + 3 of its tile, to which the 1 of I
// is added here. The chain from one
// pivot to the next is a reciprocal, a product and a multiply-add (the block's
// L D L^T); the square roots follow beside it.
template <int O>
__device__ __forceinline__ void pivot_block(Tile& T, FtSmem& sm, bool& bad) {
  const float d0 = fmaxf(1.f + tile_at(T, O, 0), 1e-30f);
  const float r0 = rcp_nr(d0);
  const float a10 = tile_at(T, O + 1, 0), a20 = tile_at(T, O + 2, 0), a30 = tile_at(T, O + 3, 0);
  const float l10 = a10 * r0, l20 = a20 * r0, l30 = a30 * r0;
  const float d1 = fmaxf(1.f + fmaf(-l10, a10, tile_at(T, O + 1, 1)), 1e-30f);
  const float a21 = fmaf(-l20, a10, tile_at(T, O + 2, 1)), a31 = fmaf(-l30, a10, tile_at(T, O + 3, 1));
  const float r1 = rcp_nr(d1);
  const float l21 = a21 * r1, l31 = a31 * r1;
  const float d2 = fmaxf(1.f + fmaf(-l21, a21, fmaf(-l20, a20, tile_at(T, O + 2, 2))), 1e-30f);
  const float a32 = fmaf(-l31, a21, fmaf(-l30, a20, tile_at(T, O + 3, 2)));
  const float r2 = rcp_nr(d2);
  const float l32 = a32 * r2;
  const float d3 =
      fmaxf(1.f + fmaf(-l32, a32, fmaf(-l31, a31, fmaf(-l30, a30, tile_at(T, O + 3, 3)))), 1e-30f);
  // a pivot that is not positive, or not finite, shows here (NaN takes 1e-30 too)
  bad |= !(fminf(fminf(d0, d1), fminf(d2, d3)) > 1e-30f) || !isfinite(d0) || !isfinite(d1) || !isfinite(d2) || !isfinite(d3);
  const float i0 = rsqrt_nr(d0), i1 = rsqrt_nr(d1), i2 = rsqrt_nr(d2), i3 = rsqrt_nr(d3);
  // the inverse of the unit lower factor, rows scaled by D^{-1/2}
  const float x20 = fmaf(l21, l10, -l20), x31 = fmaf(l32, l21, -l31);
  const float x30 = fmaf(-l32, x20, fmaf(l31, l10, -l30));
  sm.linv[0] = make_float4(i0, 0.f, 0.f, 0.f);
  sm.linv[1] = make_float4(-l10 * i1, i1, 0.f, 0.f);
  sm.linv[2] = make_float4(x20 * i2, -l21 * i2, i2, 0.f);
  sm.linv[3] = make_float4(x30 * i3, x31 * i3, -l32 * i3, i3);
}

template <int O>
__device__ __forceinline__ void leave_rows(Tile& T, FtSmem& sm, int ty) {
#pragma unroll
  for (int i = O; i < O + 4; ++i) {
    sm.raw[9 * ty + i] = tile_row(T, i);
    tile_set_row(T, i, make_float4(0.f, 0.f, 0.f, 0.f));
  }
}

// The vectors of step b = 2 p + H from their owners, and its pivot block.
template <int H>
__device__ __forceinline__ void leave_vectors(Tile& T, FtSmem& sm, int p, int ty, int cx, bool& bad) {
  const int b = 2 * p + H;
  if (cx == b && ty >= p) {
    // rows below the block; their part of the block's columns starts from 0
    if (ty > p) {
      leave_rows<0>(T, sm, ty);
      leave_rows<4>(T, sm, ty);
    } else {
      pivot_block<4 * H>(T, sm, bad);
      if (H == 0) leave_rows<4>(T, sm, ty);
    }
  } else if (ty == p && cx < b) {
#pragma unroll
    for (int v = 0; v < 4; ++v)
      sm.raw[4 * cx + (cx >> 1) + v] = make_float4(tile_at(T, 4 * H, v), tile_at(T, 4 * H + 1, v), tile_at(T, 4 * H + 2, v),
                                       tile_at(T, 4 * H + 3, v));
  }
}

// Rows O .. 7 of the tile: Z_rc -= u_r . u_c.
template <int O>
__device__ __forceinline__ void update_rows(Tile& T, const FtSmem& sm, int ty, int cx) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 c = *(const float4*)&sm.ut[j][4 * cx];
    const float2 n[4] = {make_float2(-c.x, -c.x), make_float2(-c.y, -c.y), make_float2(-c.z, -c.z),
                         make_float2(-c.w, -c.w)};
    float4 r[2];
#pragma unroll
    for (int h = O / 4; h < 2; ++h) r[h] = *(const float4*)&sm.ut[j][8 * ty + 4 * h];
#pragma unroll
    for (int h = O / 4; h < 2; ++h)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        T[2 * h][e] = __ffma2_rn(make_float2(r[h].x, r[h].y), n[e], T[2 * h][e]);
        T[2 * h + 1][e] = __ffma2_rn(make_float2(r[h].z, r[h].w), n[e], T[2 * h + 1][e]);
      }
  }
}

template <int H>
__device__ __forceinline__ void eliminate_step(Tile& T, FtSmem& sm, int p, int ty, int cx, int tid,
                                               bool& bad TRC_PARAM) {
  const int b = 2 * p + H;
  TRC_AFTER(tr_w, __float_as_int(tile_at(T, 7, 3)));
  named_barrier_sync(1, FT_THREADS);
  TRC_AFTER(tr_v, *(volatile int*)&sm.linv[3].w);
  if (tid < D) {
    const float4 m0 = sm.linv[0], m1 = sm.linv[1], m2 = sm.linv[2], m3 = sm.linv[3];
    float4 x = sm.raw[tid + (tid >> 3)];
    const int e = tid - 4 * b;  // in the block: a unit vector
    if (e >= 0 && e < 4) x = make_float4(e == 0 ? 1.f : 0.f, e == 1 ? 1.f : 0.f, e == 2 ? 1.f : 0.f, e == 3 ? 1.f : 0.f);
    const float u0 = m0.x * x.x;
    const float u1 = fmaf(m1.y, x.y, m1.x * x.x);
    const float u2 = fmaf(m2.z, x.z, fmaf(m2.y, x.y, m2.x * x.x));
    const float u3 = fmaf(m3.w, x.w, fmaf(m3.z, x.z, fmaf(m3.y, x.y, m3.x * x.x)));
    sm.ut[0][tid] = u0;
    sm.ut[1][tid] = u1;
    sm.ut[2][tid] = u2;
    sm.ut[3][tid] = u3;
  }
  named_barrier_sync(1, FT_THREADS);
  TRC_AFTER(tr_u, *(volatile int*)&sm.ut[3][D - 1]);
  if (ty >= p) {
    if (ty > p) {
      update_rows<0>(T, sm, ty, cx);
    } else {  // below the block in the tile: rows 4 .. 7 (H == 0); the block's rows are final
      if (H == 0) update_rows<4>(T, sm, ty, cx);
#pragma unroll
      for (int j = 0; j < 4; ++j) tile_set_row(T, 4 * H + j, *(const float4*)&sm.ut[j][4 * cx]);
    }
    if (H == 0) leave_vectors<1>(T, sm, p, ty, cx, bad);
    else if (p < 15) leave_vectors<0>(T, sm, p + 1, ty, cx, bad);
  }
  TRC_AFTER(tr_e, __float_as_int(tile_at(T, 7, 3)));
  if (tid == FT_TRACED) {
    TRC_SPAN(11, tr_w, tr_v);
    TRC_SPAN(12, tr_v, tr_u);
    TRC_SPAN(13, tr_u, tr_e);
  }
}

// T (the tiles of A - I) -> L^{-1}'s, by FT_THREADS threads (the last ones without a tile: ty = -1).
__device__ __forceinline__ void eliminate(Tile& T, FtSmem& sm, int ty, int cx, int tid,
                                          bool& bad TRC_PARAM) {
  if (ty >= 0) leave_vectors<0>(T, sm, 0, ty, cx, bad);
#pragma unroll 1
  for (int p = 0; p < 16; ++p) {
    eliminate_step<0>(T, sm, p, ty, cx, tid, bad TRC_PASS);
    eliminate_step<1>(T, sm, p, ty, cx, tid, bad TRC_PASS);
  }
}

// PROJ: two 128 x 128 float32 matrices, 16-byte rows.
constexpr int FT_LD = D + 4;
constexpr size_t FT_PROJ_SMEM = (size_t)2 * D * FT_LD * sizeof(float);

// acc = P Q (row-major, stride FT_LD), 8 x 8 outputs per thread of a 16 x 16 grid:
// rows 8 ty .., columns 8 tx .., from the first `mend` (a multiple of 4) columns of P
using Acc = float2[8][4];
__device__ __forceinline__ void tile_product(Acc& acc, const float* P, const float* Q, int ty, int tx, int mend = D) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int m = 0; m < mend; m += 4) {
    float2 q[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 a = *(const float4*)(Q + (m + j) * FT_LD + 8 * tx);
      const float4 b = *(const float4*)(Q + (m + j) * FT_LD + 8 * tx + 4);
      q[j][0] = make_float2(a.x, a.y), q[j][1] = make_float2(a.z, a.w);
      q[j][2] = make_float2(b.x, b.y), q[j][3] = make_float2(b.z, b.w);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 x = *(const float4*)(P + (8 * ty + i) * FT_LD + m);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        acc[i][c] = __ffma2_rn(make_float2(x.x, x.x), q[0][c], acc[i][c]);
        acc[i][c] = __ffma2_rn(make_float2(x.y, x.y), q[1][c], acc[i][c]);
        acc[i][c] = __ffma2_rn(make_float2(x.z, x.z), q[2][c], acc[i][c]);
        acc[i][c] = __ffma2_rn(make_float2(x.w, x.w), q[3][c], acc[i][c]);
      }
    }
  }
}

// T = the tile of rows 8 ty .., columns 4 cx .. of P Q, the same sums in the same order.
__device__ __forceinline__ void own_tile_product(Tile& T, const float* P, const float* Q, int ty, int cx) {
  float2 acc[8][2];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int m = 0; m < D; m += 4) {
    float4 q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) q[j] = *(const float4*)(Q + (m + j) * FT_LD + 4 * cx);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float4 x = *(const float4*)(P + (8 * ty + i) * FT_LD + m);
      const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[i][0] = __ffma2_rn(make_float2(xs[j], xs[j]), make_float2(q[j].x, q[j].y), acc[i][0]);
        acc[i][1] = __ffma2_rn(make_float2(xs[j], xs[j]), make_float2(q[j].z, q[j].w), acc[i][1]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) tile_set_row(T, i, make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y));
}

__device__ __forceinline__ void store_acc_t(const Acc& T, float* dst, int ld, int ty, int tx) {
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    auto at = [&](int i) { return (c & 1) ? T[i][c >> 1].y : T[i][c >> 1].x; };
    float* r = dst + (int64_t)(8 * tx + c) * ld + 8 * ty;
    *(float4*)r = make_float4(at(0), at(1), at(2), at(3));
    *(float4*)(r + 4) = make_float4(at(4), at(5), at(6), at(7));
  }
}

// Four consecutive values of a row as the image's hi and lo (8 bytes each).
__device__ __forceinline__ void split4(const float4 x, uint2& hi, uint2& lo) {
  hi.x = pack_bf16x2(x.x, x.y), hi.y = pack_bf16x2(x.z, x.w);
  lo.x = pack_bf16x2(x.x - bf16lo(hi.x), x.y - bf16hi(hi.x));
  lo.y = pack_bf16x2(x.z - bf16lo(hi.y), x.w - bf16hi(hi.y));
}
// Image offset of channels 4 cx .. + 3 of image row ir.
__device__ __forceinline__ uint32_t img_off(uint32_t ir, int cx) {
  return (cx >> 4) * 32768u + sw128_off(ir, (cx & 15) >> 1) + 8u * (cx & 1);
}

template <bool PROJ, int CTAS>
__global__ void __launch_bounds__(FT_THREADS, CTAS)
    factor_kernel(Dims dm, Ws ws, const float* __restrict__ out_factor, int reduced) {
  pdl_wait();
  // The one partial that the reducing launch leaves, at the unit's first chunk, read
  // without the list of partials: 0.7 us less (one layer of 4096 tokens 72.8 -> 72.1
  // us). Not with four CTAs on an SM, where the second way to read spills 38 bytes a
  // thread instead of 20 (1024 units 0.132 ms, 0.119 with the list alone; with three,
  // 26 instead of 46 bytes and 320 units 0.0576 instead of 0.0595).
  constexpr bool DIRECT = CTAS <= 3;
  extern __shared__ __align__(16) float fmat[];  // PROJ: R0, R1
  __shared__ FtSmem sm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // tile of this thread: tiles 0 .. ty (ty + 1) - 1 lie in the tile rows above ty
  int ty = (int)((sqrtf(4.f * (float)tid + 1.f) - 1.f) * 0.5f);
  while (ty * (ty + 1) > tid) --ty;
  while ((ty + 1) * (ty + 2) <= tid) ++ty;
  const int cx = tid - ty * (ty + 1);
  if (tid >= FT_TILES) ty = -1;
  const bool own = ty >= 0;
  const int u = blockIdx.x;
  const int plane = u / dm.S, s = u % dm.S;
  if (tid == 0) sm.skip = status_failed(ws) ? 1 : 0;
  const int ch0 = ws.plan[1 + s];
  const int ch1 = !DIRECT && reduced ? min(ch0 + 1, (int)ws.plan[2 + s]) : (int)ws.plan[2 + s];
  __syncthreads();
  if (sm.skip) return;
  bool bad = false;
  // time accounting (trace builds): 0 the partials summed, 8 the outputs, 9 units, 10 the
  // whole unit, 14 the products before the elimination (thread 0); of the elimination, by
  // FT_TRACED, 11 from its arrival at a step's first barrier until all vectors are left,
  // 12 from there to the second (the vectors turned into u), 13 the rest of the step
  // (update, vectors left)
  TRC_DECL(TR_CTA_SLOTS);
  TRC_T(tr_unit);

  // G's tiles: the sum of the unit's partials, in chunk order, straight from
  // global memory (layout: (m, n) at ((n / 32) D + m) 32 + n % 32)
  Tile T;
#pragma unroll
  for (int i = 0; i < 8; ++i) tile_set_row(T, i, make_float4(0.f, 0.f, 0.f, 0.f));
  {
    const float* gp = ws.gpart + ((int64_t)plane * dm.c_cap) * D * D + ((cx >> 3) * D + 8 * ty) * 32 + (cx & 7) * 4;
    const int32_t* pf = ws.pflag + (int64_t)plane * dm.c_cap;
    if (DIRECT && reduced && own && ch0 < ch1) {
      const float* src = gp + (int64_t)ch0 * D * D;
#pragma unroll
      for (int i = 0; i < 8; ++i) tile_set_row(T, i, *(const float4*)(src + i * 32));
    }
    for (int base = ch0; base < ch1 && !(DIRECT && reduced); base += FT_THREADS) {
      // the chunks that hold a partial (the first one of every run)
      const int ch = base + tid;
      const bool has = ch < ch1 && pf[ch] != 0;
      const uint32_t b = __ballot_sync(0xffffffffu, has);
      if (lane == 0) sm.cnt[warp] = __popc(b);
      __syncthreads();
      int at = 0, n = 0;
#pragma unroll
      for (int w = 0; w < FT_THREADS / 32; ++w) {
        if (w < warp) at += sm.cnt[w];
        n += sm.cnt[w];
      }
      if (has) sm.list[at + __popc(b & ((1u << lane) - 1u))] = ch;
      __syncthreads();
      if (own)
        for (int k = 0; k < n; ++k) {
          const float* src = gp + (int64_t)sm.list[k] * D * D;
          float4 v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = *(const float4*)(src + i * 32);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            tile_at(T, i, 0) += v[i].x, tile_at(T, i, 1) += v[i].y;
            tile_at(T, i, 2) += v[i].z, tile_at(T, i, 3) += v[i].w;
          }
        }
      __syncthreads();  // the list is read before the next round writes it
    }
  }
  // G, both triangles (a diagonal tile's part above the diagonal is there as it is)
  if (own) {
    float* gout = ws.gram + (int64_t)u * D * D;
#pragma unroll
    for (int i = 0; i < 8; ++i) *(float4*)(gout + (8 * ty + i) * D + 4 * cx) = tile_row(T, i);
    if (cx < 2 * ty) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float* r = gout + (4 * cx + c) * D + 8 * ty;
        *(float4*)r = make_float4(tile_at(T, 0, c), tile_at(T, 1, c), tile_at(T, 2, c), tile_at(T, 3, c));
        *(float4*)(r + 4) = make_float4(tile_at(T, 4, c), tile_at(T, 5, c), tile_at(T, 6, c), tile_at(T, 7, c));
      }
    }
  }
  TRC_AFTER(tr_g, __float_as_int(tile_at(T, 0, 0)));
  if (tid == 0) {
    TRC_SPAN(0, tr_unit, tr_g);
    TRC_INC(9);
  }
  float *R0 = fmat, *R1 = fmat + D * FT_LD;
  const int py = tid >> 4, px = tid & 15;  // the products' grid (threads 0-255)
  if constexpr (PROJ) {
    TRC_T(tr_p);
    // M = F G F^T: (F G)^T to R0, then the tiles of M = F (F G)^T (M is symmetric)
    const float* F = out_factor + (int64_t)plane * D * D;
    if (own) {
#pragma unroll
      for (int i = 0; i < 8; ++i) *(float4*)(R0 + (8 * ty + i) * FT_LD + 4 * cx) = tile_row(T, i);
      if (cx < 2 * ty) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float* r = R0 + (4 * cx + c) * FT_LD + 8 * ty;
          *(float4*)r = make_float4(tile_at(T, 0, c), tile_at(T, 1, c), tile_at(T, 2, c), tile_at(T, 3, c));
          *(float4*)(r + 4) = make_float4(tile_at(T, 4, c), tile_at(T, 5, c), tile_at(T, 6, c), tile_at(T, 7, c));
        }
      }
    }
    for (int e = tid; e < D * D / 4; e += FT_THREADS)
      *(float4*)(R1 + (e >> 5) * FT_LD + (e & 31) * 4) = ((const float4*)F)[e];
    Acc acc;
    __syncthreads();
    if (tid < 256) tile_product(acc, R1, R0, py, px);
    __syncthreads();
    if (tid < 256) store_acc_t(acc, R0, FT_LD, py, px);
    __syncthreads();
    if (own) own_tile_product(T, R1, R0, ty, cx);
    __syncthreads();
    if (tid == 0) TRC_ADD(14, tr_p);
  }
  eliminate(T, sm, ty, cx, tid, bad TRC_PASS);
  TRC_T(tr_o);
  if (own && cx >= 2 * ty) {  // zeros above the diagonal
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (4 * (cx - 2 * ty) + c > i) tile_at(T, i, c) = 0.f;
  }
  float* mout = ws.minv + (int64_t)u * D * D;
  uint8_t* img = ws.minv_img + (int64_t)u * 65536;
  if constexpr (PROJ) {  // T = L_M^{-1} F
    for (int e = tid; e < D * D / 4; e += FT_THREADS) {  // the tiles above the diagonal
      const int r = e >> 5, c4 = e & 31;
      if (c4 > 2 * (r >> 3) + 1) *(float4*)(R0 + r * FT_LD + 4 * c4) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (own) {
#pragma unroll
      for (int i = 0; i < 8; ++i) *(float4*)(R0 + (8 * ty + i) * FT_LD + 4 * cx) = tile_row(T, i);
    }
    __syncthreads();
    if (tid < 256) {
      // L_M^{-1}'s rows end at the diagonal: the 16 rows of a warp need as many
      // columns as its last row has; warps w and w + 4, which share a sub-partition,
      // take the row blocks w and 7 - w, i.e. 144 columns between them
      Acc acc;
      const int pr = py < 8 ? py : 23 - py;
      tile_product(acc, R0, R1, pr, px, 16 * ((pr >> 1) + 1));
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t n = 8 * pr + i;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 x = make_float4(acc[i][2 * h].x, acc[i][2 * h].y, acc[i][2 * h + 1].x, acc[i][2 * h + 1].y);
          bad |= !isfinite(x.x) || !isfinite(x.y) || !isfinite(x.z) || !isfinite(x.w);
          *(float4*)(mout + n * D + 8 * px + 4 * h) = x;
          uint2 hi, lo;
          split4(x, hi, lo);
          *(uint2*)(img + img_off(n, 2 * px + h)) = hi;
          *(uint2*)(img + img_off(n + 128, 2 * px + h)) = lo;
        }
      }
    }
  } else {
    if (own) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t n = 8 * ty + i;
        const float4 x = tile_row(T, i);
        bad |= !isfinite(x.x) || !isfinite(x.y) || !isfinite(x.z) || !isfinite(x.w);
        *(float4*)(mout + n * D + 4 * cx) = x;
        uint2 hi, lo;
        split4(x, hi, lo);
        const uint32_t ir = 32 * (n >> 4) + (n & 15);
        *(uint2*)(img + img_off(ir, cx)) = hi;
        *(uint2*)(img + img_off(ir + 16, cx)) = lo;
      }
    }
    // zeros: float32 above the tiles; in the image the score pass reads row n up
    // to channel 16 (n / 16) + 15, so only the tile pair right of an even tile row
    for (int e = tid; e < D * D / 4; e += FT_THREADS) {
      const int r = e >> 5, c4 = e & 31, t = r >> 3;
      if (c4 <= 2 * t + 1) continue;
      *(float4*)(mout + r * D + 4 * c4) = make_float4(0.f, 0.f, 0.f, 0.f);
      if ((t & 1) == 0 && c4 <= 2 * t + 3) {
        const uint32_t ir = 32 * (r >> 4) + (r & 15);
        *(uint2*)(img + img_off(ir, c4)) = make_uint2(0u, 0u);
        *(uint2*)(img + img_off(ir + 16, c4)) = make_uint2(0u, 0u);
      }
    }
  }
  if (tid == 0) {
    TRC_ADD(8, tr_o);
    TRC_ADD(10, tr_unit);
  }
  if (tid == 0 || tid == FT_TRACED) TRC_PUT(ws, TR_K_FACTOR, TR_CTA_SLOTS);
  if (bad) flag(ws, ST_NONFINITE);
}

// The partials of each unit summed into the first one (at its first chunk), by
// one CTA per unit and lower 32 x 32 block: for a few units with many partials,
// which the factor's one CTA per unit would add one after the other (~0.6 us each;
// this launch costs about 4 us, hence from six partials on, by the mean over the
// units: a long request beside many short ones may keep some twenty for the factor).
constexpr int FR_THREADS = 256;
__global__ void __launch_bounds__(FR_THREADS) gram_reduce_kernel(Dims dm, Ws ws) {
  pdl_wait();
  __shared__ int s_skip;
  const int tid = threadIdx.x;
  if (tid == 0) s_skip = status_failed(ws) ? 1 : 0;
  const int u = blockIdx.x / 10, blk = blockIdx.x % 10;
  const int nb = blk < 4 ? 0 : (blk < 7 ? 1 : (blk < 9 ? 2 : 3));             // column block
  const int I = nb + blk - (nb == 0 ? 0 : (nb == 1 ? 4 : (nb == 2 ? 7 : 9)));  // row block >= nb
  const int plane = u / dm.S, s = u % dm.S;
  const int ch0 = ws.plan[1 + s], ch1 = ws.plan[2 + s];
  __syncthreads();
  if (s_skip || ch0 >= ch1) return;
  float* gp = ws.gpart + ((int64_t)plane * dm.c_cap) * D * D + (nb * D + 32 * I) * 32 + 4 * tid;
  const int32_t* pf = ws.pflag + (int64_t)plane * dm.c_cap;
  float4 acc = *(const float4*)(gp + (int64_t)ch0 * D * D);
  __shared__ int s_list[FR_THREADS], s_cnt[FR_THREADS / 32];
  const int lane = tid & 31, warp = tid >> 5;
  for (int base = ch0 + 1; base < ch1; base += FR_THREADS) {
    // the chunks that hold a partial
    const bool has = base + tid < ch1 && pf[base + tid] != 0;
    const uint32_t b = __ballot_sync(0xffffffffu, has);
    __syncthreads();
    if (lane == 0) s_cnt[warp] = __popc(b);
    __syncthreads();
    int at = 0, n = 0;
#pragma unroll
    for (int w = 0; w < FR_THREADS / 32; ++w) {
      if (w < warp) at += s_cnt[w];
      n += s_cnt[w];
    }
    if (has) s_list[at + __popc(b & ((1u << lane) - 1u))] = base + tid;
    __syncthreads();
    constexpr int N = 16;  // loads in flight
    for (int k0 = 0; k0 < n; k0 += N) {
      float4 v[N];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k0 + k < n) v[k] = *(const float4*)(gp + (int64_t)s_list[k0 + k] * D * D);
      }
#pragma unroll
      for (int k = 0; k < N; ++k) acc.x += v[k].x, acc.y += v[k].y, acc.z += v[k].z, acc.w += v[k].w;
    }
  }
  *(float4*)(gp + (int64_t)ch0 * D * D) = acc;
}

cudaError_t launch_factor(const Dims& dm, const Ws& ws, const float* out_factor, int partials, int sms,
                          cudaStream_t st) {
  const int units = dm.L * dm.Hkv * dm.S;
  const int reduced = partials >= 6 ? 1 : 0;
  if (reduced) JACAP_TRY(launch_pdl(dm.pdl != 0, gram_reduce_kernel, units * 10, FR_THREADS, 0, st, dm, ws));
  if (out_factor != nullptr) {
    auto kern = factor_kernel<true, 1>;
    JACAP_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FT_PROJ_SMEM));
    JACAP_TRY(launch_pdl(dm.pdl != 0, kern, units, FT_THREADS, FT_PROJ_SMEM, st, dm, ws, out_factor, reduced));
  } else {
    // CTAs per SM (2, 3 or 4; with 96, 72 or 56 registers a thread): more of them
    // finish more units in the same time but each later, and all units of a round
    // end together, so the choice is the least rounds x time of a round in us (256
    // units: 38 with two; 448: 55 with three, 65 with two; 1024: 115 with four, 128
    // with three, 150 with two)
    constexpr int ROUND_US[3] = {38, 50, 58};
    int best = 0;
    for (int i = 0; i < 3; ++i) {
      auto cost = [&](int k) { return (int64_t)((units + (k + 2) * sms - 1) / ((k + 2) * sms)) * ROUND_US[k]; };
      if (cost(i) < cost(best)) best = i;
    }
    auto kern = best == 0 ? factor_kernel<false, 2> : (best == 1 ? factor_kernel<false, 3> : factor_kernel<false, 4>);
    JACAP_TRY(launch_pdl(dm.pdl != 0, kern, units, FT_THREADS, 0, st, dm, ws, out_factor, reduced));
  }
  return cudaGetLastError();
}

}  // namespace jacap
