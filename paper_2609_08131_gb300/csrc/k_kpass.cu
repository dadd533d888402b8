// k_kpass.cu - streaming K pass for bf16 caches.
//
// For every token i of a unit and every query head h of its GQA group:
//   l_h,i     = k_i . mu_h / (tau sqrt d)      pool-softmax logit (Sec. 3.4; Alg. 1 step 1)
//   kappa_h,i = sum_c lambda_h,c k_i,c^2       diagonal query-response variance (Sec. 3.4)
// plus an online (max, sum exp(l - max)) per work item and head, which the
// weight pass combines into the softmax normaliser.
//
// Both are 128 x 128 x N contractions per 128-token tile and run on the tensor
// cores. The logits take the TMA-staged K tile as A and B = mu' = mu / (tau sqrt
// d); kappa takes the tile's squares, k^2 = hi + lo with hi = RN_bf16(k^2) and lo
// = k^2 - hi (exact: a bf16 square has 16 significant bits; one packed multiply
// and one packed fused multiply-add give both), which the convert warps write
// into tensor memory as two A operands (lane = token, two channels per column),
// and B = lambda. mu' and lambda are split exactly into three bf16 parts (hi +
// mid + lo carries ~24 significant bits) for the G heads, so the products are
// those of float32 operands (k^2 while its lo part is not subnormal: |k| > 2^-58).
//
// The MMAs' fp32 sums truncate, which would leave kappa's sums of positive terms too
// small by half a unit in the last place per addition. So kappa's K-steps go into KG
// groups of columns (four of 2 steps; three of 3, 3 and 2 for G > 5, where a group
// takes twice the columns) that the readout adds, and the sum is recentred: of m
// additions of about equal terms the j-th truncates at a sum of j / m of the group's,
// losing 2^-24 / (2 ln 2) of it on average over a mantissa, together (m + 1) 2^-23 /
// (8 ln 2) of the group's sum, which the readout adds to the small parts before its
// last addition rounds. Error of sum_h kappa against 64 bits, rms (n = 8192, windows of
// 32): 4.8e-8, 4.5e-8, 4.6e-8, 5.0e-8, 5.1e-8 for G = 1, 4, 5, 7, 8, and 4.8e-8, 4.5e-8,
// 4.6e-8, 4.9e-8, 5.0e-8 with float32 multiply-adds; not recentred (two groups for G >
// 5) 8.0e-8, 7.7e-8, 7.8e-8, 1.27e-7, 1.27e-7. With four key channels 8 times the others
// 5.2e-8, 4.8e-8, 4.9e-8, 5.3e-8, 5.5e-8 (multiply-adds 5.2e-8, 4.6e-8, 4.7e-8, 5.0e-8,
// 5.1e-8). Recentring costs no time, the third group 1 % of the K pass at G = 7 and 8.
// The softmax sums take expf: with __expf they were 3.4e-8 too small and the weights
// 9e-8 too large (n >= 32768), with it 0.3e-8 to 0.8e-8 and 1.5e-8 to 2.8e-8.
//
// Why this way: issued under elect.sync, an M = 128, N = 16 MMA costs 9 cycles
// with A in tensor memory and 39 with A in shared memory (45 either way under a
// lane test), so a tile's 24 MMAs take ~460 of the ~1500 cycles in which its 32
// KB arrive at the copy rate. On the CUDA cores kappa took 1.2 us per tile and
// group of four warps at G = 4, and grew with G. Measured, both kinds, K pass
// alone (events): 32 layers x 8 KV heads x 32768 tokens, G = 4: 0.403 -> 0.385
// ms; 40 x 8 x 9001, G = 5: 0.202 -> 0.147 ms; 28 x 4 x 20011, G = 7: 0.209 ->
// 0.136 ms; and with the runs dealt as CTAs become free (RunStream) 0.352, 0.137
// and 0.122 ms. What bounds it now is HBM (6.9 TB/s of K and rows at G = 4).
//
// Warp roles: 0 TMA producer; 1 issues the MMAs; 2 builds the mu' and lambda
// images of each unit a CTA reaches (double-buffered, one run of the unit's
// consecutive items ahead); 3-10 convert (two warps per tensor-memory lane
// quarter, each 32 tokens x 64 channels); 11-14 read the accumulators back (one
// lane quarter each), keep the online softmax statistics and store each token's
// row (logits, kappa) in one piece.
#include "jacap_dev.cuh"
#include "jacap_internal.h"

namespace jacap {

constexpr int KB_BOX = 16384;    // {64 channels, 128 tokens} bf16
constexpr int KB_TILE_BYTES = 2 * KB_BOX;
constexpr int KB_THREADS = 480;
constexpr int KB_BUILD_WARP = 2, KB_CONV_WARP0 = 3, KB_CONV_WARPS = 8, KB_READ_WARP0 = 11;
constexpr uint32_t KB_TMEM_COLS = 512;
constexpr uint32_t KB_ACC_COLS = 256;  // columns [0, 256): accumulators
constexpr uint32_t KB_A_COLS = 128;    // an A buffer: hi(k^2) [0, 64), lo(k^2) [64, 128)
static_assert(KB_ACC_COLS + 2 * KB_A_COLS <= KB_TMEM_COLS, "tensor memory budget");

template <int G>
struct KbCfg {
  static constexpr int NB = (3 * G <= 16) ? 16 : 32;  // MMA N = rows of an image
  static constexpr int KG = NB == 16 ? 4 : 3;          // kappa's channel groups, each with columns of its own
  static constexpr int step0(int g) { return (g * (D / 16) + KG - 1) / KG; }  // K-steps (16 channels) before group g
  // what truncation takes from kappa on average, relative (see the top)
  static constexpr float recentre() {
    float c = 0.f;
    for (int g = 0; g < KG; ++g) {
      const int m = step0(g + 1) - step0(g);
      c += (float)m / (D / 16) * (float)(m + 1) * 0.18033688f;  // 1 / (8 ln 2)
    }
    return c * 1.1920929e-7f;  // 2^-23
  }
  static constexpr int ACC = (1 + KG) * NB;            // columns of an accumulator slot: logits, then the groups
  static constexpr int NACC = KB_ACC_COLS / ACC;
  static constexpr int IMG_ATOM = NB * 128;            // bytes per 64-channel atom
  static constexpr int IMG_BYTES = 2 * IMG_ATOM;       // one image; a run has two (mu', lambda)
  static constexpr uint32_t IDESC = idesc_bf16_f32(128, NB, 0, 0);
  static constexpr size_t smem_for(int stages) {
    return 1024 + (size_t)stages * KB_TILE_BYTES + 4 * IMG_BYTES + TILE * 2 * G * 4 + 8 * 2 * G * 4 + 256;  // + barriers
  }
  static constexpr int STAGES = smem_for(6) + 512 <= 232448 ? 6 : 5;  // K tiles in flight
  static constexpr size_t SMEM = smem_for(STAGES);
};

// The images of one run: row n = part G + h of an image holds part (0 hi, 1 mid,
// 2 lo) of mu'_h (image 0) or lambda_h (image 1), K-major with the 128-byte
// swizzle (two 64-channel atoms). Each lane takes 8 channels of a head at a
// time: one read of the values gives all three parts (rows 3 G .. NB - 1 stay
// zero).
template <int G>
__device__ __forceinline__ void build_split_images(uint8_t* im, const float* mu, const float* lam, int lane) {
  using C = KbCfg<G>;
  constexpr int NB2 = G <= 2 ? 1 : 2;  // values of this many turns are loaded together
#pragma unroll 1
  for (int e0 = lane; e0 < G * 16; e0 += 32 * NB2) {
    float4 v[NB2][4];
#pragma unroll
    for (int i = 0; i < NB2; ++i) {
      const int e = e0 + 32 * i;
      if (e < G * 16) {
        v[i][0] = *(const float4*)(mu + e * 8);
        v[i][1] = *(const float4*)(mu + e * 8 + 4);
        v[i][2] = *(const float4*)(lam + e * 8);
        v[i][3] = *(const float4*)(lam + e * 8 + 4);
      }
    }
#pragma unroll
    for (int i = 0; i < NB2; ++i) {
      const int e = e0 + 32 * i, h = e >> 4, cc = e & 15;
      if (e >= G * 16) break;
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const float4 p = v[i][2 * m], q = v[i][2 * m + 1];
        const float x[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
        uint32_t w[3][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          w[0][j] = pack_bf16x2(x[2 * j], x[2 * j + 1]);
          const float r0 = x[2 * j] - bf16lo(w[0][j]), r1 = x[2 * j + 1] - bf16hi(w[0][j]);
          w[1][j] = pack_bf16x2(r0, r1);
          w[2][j] = pack_bf16x2(r0 - bf16lo(w[1][j]), r1 - bf16hi(w[1][j]));
        }
#pragma unroll
        for (int part = 0; part < 3; ++part)
          *(uint4*)(im + m * C::IMG_BYTES + (cc >> 3) * C::IMG_ATOM + sw128_off(part * G + h, cc & 7)) =
              make_uint4(w[part][0], w[part][1], w[part][2], w[part][3]);
      }
    }
  }
}

template <int G>
__global__ void __launch_bounds__(KB_THREADS, 1)
    kpass_bf16_kernel(const __grid_constant__ CUtensorMap kmap, Dims dm, Ws ws, const int32_t* __restrict__ cu) {
  pdl_wait();
  using C = KbCfg<G>;
  constexpr int KB_STAGES = C::STAGES, NACC = C::NACC, NB = C::NB;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* tiles = smem;
  uint8_t* img = tiles + KB_STAGES * KB_TILE_BYTES;  // [parity][mu', lambda][IMG_BYTES]
  float* rows = (float*)(img + 4 * C::IMG_BYTES);     // [TILE][2G] the tile's rows on their way out
  float* red = rows + TILE * 2 * G;                   // [run parity][4 readout warps][2G]
  uint64_t* full = (uint64_t*)(red + 8 * 2 * G);
  uint64_t* empty = full + KB_STAGES;
  uint64_t* afull = empty + KB_STAGES;   // [2] the tile's A operands are in tensor memory
  uint64_t* aempty = afull + 2;          // [2] the MMAs have read them
  uint64_t* accfull = aempty + 2;        // [NACC]
  uint64_t* accempty = accfull + NACC;   // [NACC]
  uint64_t* imgready = accempty + NACC;  // [2]
  uint64_t* imgfree = imgready + 2;      // [2]
  static_assert((2 * KB_STAGES + 4 + 2 * NACC + 4) * 8 <= 256, "barriers");
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort, s_skip;
  __shared__ RunQueue s_queue;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    s_abort = 0;
    s_skip = status_failed(ws) ? 1 : 0;
    run_queue_init(&s_queue, 2 + KB_CONV_WARPS + 4);  // MMA, builder, convert and readout warps
    for (int i = 0; i < KB_STAGES; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), KB_CONV_WARPS + 1);  // and the MMAs' commit
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&afull[i]), KB_CONV_WARPS);
      mbar_init(smem_u32(&aempty[i]), 1);
      mbar_init(smem_u32(&imgready[i]), 1);
      mbar_init(smem_u32(&imgfree[i]), 1);
    }
    for (int i = 0; i < NACC; ++i) {
      mbar_init(smem_u32(&accfull[i]), 1);
      mbar_init(smem_u32(&accempty[i]), 4);
    }
    fence_mbar_init();
  }
  for (int e = tid; e < 4 * C::IMG_BYTES / 16; e += KB_THREADS) ((uint4*)img)[e] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  __syncthreads();
  if (s_skip) return;
  if (warp == 1) {
    tmem_alloc(smem_u32(&s_tmem), KB_TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  volatile int* abort = &s_abort;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer --------
    if (lane == 0) {
      prefetch_tmap(&kmap);
      uint32_t it = 0;
      bool ok = true;
      Item item;
      // time accounting (trace builds): 0 waits for a free stage, 1 the whole loop
      TRC_DECL(TR_CTA_SLOTS);
      TRC_T(tr_all);
      for (RunStream<true> is(dm, ws, &s_queue, abort, true, SCHED_KPASS); ok && is.next(item);) {
        const int l = item.plane / dm.Hkv, g = item.plane % dm.Hkv;
        for (int64_t t = item.t0; t < item.t1; t += TILE) {
          const int st = it % KB_STAGES;
          TRC_T(tr_w);
          if (it >= (uint32_t)KB_STAGES &&
              !mbar_wait(smem_u32(&empty[st]), ((it / KB_STAGES) & 1) ^ 1, ws, abort)) {
            ok = false;
            break;
          }
          TRC_ADD(0, tr_w);
          uint8_t* kt = tiles + st * KB_TILE_BYTES;
          const uint32_t fb = smem_u32(&full[st]);
          mbar_arrive_expect_tx(fb, KB_TILE_BYTES);
          tma_load_4d(smem_u32(kt), &kmap, 0, (int)t, g, l, fb);
          tma_load_4d(smem_u32(kt + KB_BOX), &kmap, 64, (int)t, g, l, fb);
          ++it;
        }
      }
      TRC_ADD(1, tr_all);
      TRC_PUT(ws, TR_K_KPASS, 2);
      for (uint32_t k = (it > (uint32_t)KB_STAGES ? it - KB_STAGES : 0); k < it; ++k)
        mbar_wait(smem_u32(&full[k % KB_STAGES]), (k / KB_STAGES) & 1, ws, nullptr);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer ----------
    if (elect_one()) {
      uint32_t it = 0, nrun = 0;  // nrun: runs of consecutive items of one unit started
      bool ok = true, cont = false;
      int p = 0;
      Item item;
      // time accounting (trace builds): 2 waits for an image, 3 for a tile's operands and a
      // free accumulator, 5 the whole loop, 6 tiles
      TRC_DECL(TR_CTA_SLOTS);
      TRC_T(tr_all);
      for (RunStream<false> is(dm, ws, &s_queue, abort, true); ok && is.next(item);) {
        if (!cont) {
          p = nrun & 1;
          TRC_T(tr_i);
          if (!mbar_wait(smem_u32(&imgready[p]), (nrun >> 1) & 1, ws, abort)) break;
          TRC_ADD(2, tr_i);
          tc_fence_after();
        }
        const uint64_t bmu = smem_desc_sw128(smem_u32(img + (2 * p) * C::IMG_BYTES), 16, 1024);
        const uint64_t blam = smem_desc_sw128(smem_u32(img + (2 * p + 1) * C::IMG_BYTES), 16, 1024);
        for (int64_t t = item.t0; t < item.t1; t += TILE, ++it) {
          const int ab = it & 1, ac = it % NACC;
          TRC_T(tr_f);
          const int st = it % KB_STAGES;
          if (!mbar_wait(smem_u32(&full[st]), (it / KB_STAGES) & 1, ws, abort) ||
              !mbar_wait(smem_u32(&afull[ab]), (it >> 1) & 1, ws, abort) ||
              (it >= (uint32_t)NACC && !mbar_wait(smem_u32(&accempty[ac]), ((it / NACC) & 1) ^ 1, ws, abort))) {
            ok = false;
            break;
          }
          TRC_ADD(3, tr_f);
          TRC_INC(6);
          tc_fence_after();
          // descriptors advance by (byte offset >> 4) in their address field
          const uint32_t a = tmem + KB_ACC_COLS + ab * KB_A_COLS;
          const uint64_t a0 = smem_desc_sw128(smem_u32(tiles + st * KB_TILE_BYTES), 16, 1024);
          const uint32_t dl = tmem + ac * C::ACC;
#pragma unroll
          for (int g = 0; g < C::KG; ++g) {
#pragma unroll
            for (int part = 0; part < 2; ++part)  // lo first: the sums stay small until the last steps
#pragma unroll
              for (int k = C::step0(g); k < C::step0(g + 1); ++k)
                umma_f16_ts(dl + (1 + g) * NB, a + (part == 0 ? 64 : 0) + 8 * k,
                            blam + (uint64_t)((((k >> 2) * C::IMG_ATOM) + (k & 3) * 32) >> 4), C::IDESC,
                            part == 0 && k == C::step0(g) ? 0u : 1u);
          }
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
            umma_f16_ss(dl, a0 + (uint64_t)((((k >> 2) * KB_BOX) + (k & 3) * 32) >> 4),
                        bmu + (uint64_t)((((k >> 2) * C::IMG_ATOM) + (k & 3) * 32) >> 4), C::IDESC, k > 0 ? 1u : 0u);
          umma_commit(smem_u32(&empty[st]));
          umma_commit(smem_u32(&aempty[ab]));
          umma_commit(smem_u32(&accfull[ac]));
        }
        if (!ok) break;
        cont = is.next_same_unit(item);
        if (!cont) {
          umma_commit(smem_u32(&imgfree[p]));
          ++nrun;
        }
      }
      // every MMA issued here completes before the CTA tears down tensor memory
      if (it > 0) mbar_wait(smem_u32(&accfull[(it - 1) % NACC]), ((it - 1) / NACC) & 1, ws, nullptr);
      TRC_ADD(5, tr_all);
      TRC_PUT(ws, TR_K_KPASS, 7);
    }
  } else if (warp == KB_BUILD_WARP) {
    // ------------------ mu' and lambda images, once per run, one run ahead
    uint32_t nrun = 0;
    bool cont = false;
    Item item;
    for (RunStream<false> is(dm, ws, &s_queue, abort, false); is.next(item);) {
      const bool same = cont;
      cont = is.next_same_unit(item);
      if (same) continue;  // the run's images are in place
      const int l = item.plane / dm.Hkv, g = item.plane % dm.Hkv;
      const int p = nrun & 1;
      if (nrun >= 2 && !mbar_wait(smem_u32(&imgfree[p]), ((nrun >> 1) - 1) & 1, ws, abort)) break;
      const int64_t qb = (((int64_t)item.seq * dm.L + l) * dm.Hq + (int64_t)g * G) * D;
      build_split_images<G>(img + 2 * p * C::IMG_BYTES, ws.mu + qb, ws.lam + qb, lane);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&imgready[p]));
      ++nrun;
    }
  } else if (warp >= KB_CONV_WARP0 && warp < KB_CONV_WARP0 + KB_CONV_WARPS) {
    // ------------------------------------------------ convert -------------
    // Lane = token 32 quarter + lane of the tile, 64 channels of it: 128 bytes
    // from the staged tile (eight 16-byte loads, free of bank conflicts under
    // the swizzle), 32 columns of each of the three operands.
    const int quarter = warp & 3, half = (warp - KB_CONV_WARP0) >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    uint32_t it = 0;
    Item item;
    // time accounting (trace builds, first convert warp): 7 waits for a K tile, 8 for a
    // free operand buffer, 9 the conversion, 11 the loop
    TRC_DECL(TR_CTA_SLOTS);
    TRC_T(tr_all);
    // Every wait is bounded and the warps meet at no named barrier, so a warp
    // whose wait failed (the abort flag is set) leaves on its own.
    for (RunStream<false> is(dm, ws, &s_queue, abort, false); is.next(item);) {
      for (int64_t t = item.t0; t < item.t1; t += TILE, ++it) {
        const int st = it % KB_STAGES, ab = it & 1;
        TRC_T(tr_f);
        if (!mbar_wait(smem_u32(&full[st]), (it / KB_STAGES) & 1, ws, abort)) goto conv_done;
        TRC_ADD(7, tr_f);
        const uint32_t kt = smem_u32(tiles + st * KB_TILE_BYTES + half * KB_BOX);
        uint32_t r[32];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const uint4 v = lds_u128(kt + sw128_off(row, c));
          r[4 * c] = v.x, r[4 * c + 1] = v.y, r[4 * c + 2] = v.z, r[4 * c + 3] = v.w;
        }
        uint32_t hi[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) hi[c] = bf16x2_mul(r[c], r[c]);
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&empty[st]));  // the tile is in registers
        TRC_T(tr_a);
        if (it >= 2 && !mbar_wait(smem_u32(&aempty[ab]), ((it >> 1) & 1) ^ 1, ws, abort)) goto conv_done;
        TRC_ADD(8, tr_a);
        TRC_T(tr_b);
        tc_fence_after();
        const uint32_t a = tmem + KB_ACC_COLS + ab * KB_A_COLS + 32 * half + lanes;
        tmem_st_32x32b_x32(a, hi);
#pragma unroll
        for (int c = 0; c < 32; ++c) r[c] = bf16x2_fma(r[c], r[c], bf16x2_neg(hi[c]));  // lo, exact
        tmem_st_32x32b_x32(a + 64, r);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&afull[ab]));
        TRC_ADD(9, tr_b);
      }
    }
  conv_done:
    TRC_ADD(11, tr_all);
    if (warp == KB_CONV_WARP0 && lane == 0) TRC_PUT(ws, TR_K_KPASS, 12);
  } else if (warp >= KB_READ_WARP0) {
    // ------------------------------------------------ readout + stats -----
    const int quarter = warp & 3;
    const int y = quarter * 32 + lane;        // token row (tensor-memory lane)
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    const int rw = warp - KB_READ_WARP0;
    uint32_t it = 0;
    bool bad = false, cont = false;
    int par = 0;
    float run_m[G], run_s[G];
    Item item;
    // time accounting (trace builds, first readout warp): 12 waits for an accumulator, 13
    // the readout of a tile, 14 the whole loop
    TRC_DECL(TR_CTA_SLOTS);
    TRC_T(tr_all);
    for (RunStream<false> is(dm, ws, &s_queue, abort, false);;) {
      if (!is.next(item)) {  // no more runs, or a failed wait: the four warps leave together (see below)
        named_barrier_any(1, 128, is.failed);
        break;
      }
      if (!cont) {  // a new run of the unit's consecutive chunks: fresh statistics
#pragma unroll
        for (int h = 0; h < G; ++h) {
          run_m[h] = -INFINITY;
          run_s[h] = 0.f;
        }
      }
      float* lkp = ws.lk + (int64_t)item.plane * dm.Ntot * (2 * G);
      for (int64_t t = item.t0; t < item.t1; t += TILE, ++it) {
        const int ac = it % NACC;
        TRC_T(tr_f);
        if (!mbar_wait(smem_u32(&accfull[ac]), (it / NACC) & 1, ws, abort)) break;  // abort: see below
        TRC_ADD(12, tr_f);
        TRC_T(tr_b);
        tc_fence_after();
        // NB columns of logit parts, then NB of kappa parts per channel group:
        // part p of head h in column p G + h
        const uint32_t src = tmem + ac * C::ACC + lanes;
        float row[2 * G];  // logits, then kappa; the small parts first
        {
          constexpr int PS = NB == 16 ? G : 8;  // part p of head h at dv[p PS + h]
          float dv[NB == 16 ? 16 : 24];
          auto load = [&](uint32_t col) {
            if constexpr (NB == 16) tmem_ld16(col, dv);
            else tmem_ld8x3(col, G, dv);
          };
          float low[G];
          load(src);
#pragma unroll
          for (int h = 0; h < G; ++h) row[h] = dv[h] + (dv[PS + h] + dv[2 * PS + h]);
#pragma unroll
          for (int g = 1; g <= C::KG; ++g) {
            load(src + g * NB);
#pragma unroll
            for (int h = 0; h < G; ++h) {
              row[G + h] = g == 1 ? dv[h] : row[G + h] + dv[h];
              low[h] = g == 1 ? dv[PS + h] + dv[2 * PS + h] : low[h] + (dv[PS + h] + dv[2 * PS + h]);
            }
          }
#pragma unroll
          for (int h = 0; h < G; ++h) row[G + h] += fmaf(C::recentre(), row[G + h], low[h]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&accempty[ac]));
        if (t + y < item.t1) {
#pragma unroll
          for (int h = 0; h < G; ++h) {
            const float lg = row[h];
            bad |= !isfinite(lg) || !isfinite(row[G + h]);
            // branch-free online update: one of the two exponentials is exp(0)
            const float mn = fmaxf(run_m[h], lg);
            run_s[h] = run_s[h] * expf(run_m[h] - mn) + expf(lg - mn);
            run_m[h] = mn;
          }
        }
        store_rows<G>(lkp, rows, row, t, item.t1, quarter, lane);
        TRC_ADD(13, tr_b);
      }
      // ---- softmax statistics of a run, at its last chunk; the run's other
      // chunks get empty statistics (m = -inf, s = 0), which merge as nothing
      cont = is.next_same_unit(item);
      if (cont) {
        if (rw == 0 && lane < G) {
          float* cs = ws.cstats + (((int64_t)item.plane * dm.c_cap + item.cidx) * G + lane) * 2;
          cs[0] = -INFINITY;
          cs[1] = 0.f;
        }
        continue;
      }
#pragma unroll
      for (int h = 0; h < G; ++h) {
        softmax_warp_merge(run_m[h], run_s[h]);
        if (lane == 0) {
          red[(par * 4 + rw) * 2 * G + h] = run_m[h];
          red[(par * 4 + rw) * 2 * G + G + h] = run_s[h];
        }
      }
      // One barrier per run, and one before leaving: a warp that met an abort, or
      // could not take its next run, still arrives at it; the barrier ORs the
      // flag, so all four leave together.
      if (named_barrier_any(1, 128, *abort != 0)) goto read_done;
      if (rw == 0 && lane < G) {
        const int h = lane;
        float m = -INFINITY, ssum = 0.f;
        for (int j = 0; j < 4; ++j)
          softmax_merge(m, ssum, red[(par * 4 + j) * 2 * G + h], red[(par * 4 + j) * 2 * G + G + h]);
        float* cs = ws.cstats + (((int64_t)item.plane * dm.c_cap + item.cidx) * G + h) * 2;
        cs[0] = m;
        cs[1] = ssum;
      }
      par ^= 1;  // the next run's partials go elsewhere: no second barrier
    }
  read_done:
    TRC_ADD(14, tr_all);
    if (warp == KB_READ_WARP0 && lane == 0) TRC_PUT(ws, TR_K_KPASS, 15);
    if (bad) flag(ws, ST_NONFINITE);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, KB_TMEM_COLS);
  }
}

template <int G>
static cudaError_t launch_g(const CUtensorMap& kmap, const Dims& dm, const Ws& ws, const int32_t* cu, int grid,
                            cudaStream_t st) {
  constexpr size_t smem = KbCfg<G>::SMEM;
  static_assert(smem + 512 <= 232448, "shared memory budget");  // 512: the static variables
  cudaError_t e = cudaFuncSetAttribute(kpass_bf16_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  JACAP_TRY(launch_pdl(dm.pdl != 0, kpass_bf16_kernel<G>, grid, KB_THREADS, smem, st, kmap, dm, ws, cu));
  return cudaGetLastError();
}

cudaError_t launch_kpass_bf16(const CUtensorMap& kmap, const Dims& dm, const Ws& ws, const int32_t* cu, int grid,
                              cudaStream_t st) {
  switch (dm.G) {
    case 1: return launch_g<1>(kmap, dm, ws, cu, grid, st);
    case 2: return launch_g<2>(kmap, dm, ws, cu, grid, st);
    case 3: return launch_g<3>(kmap, dm, ws, cu, grid, st);
    case 4: return launch_g<4>(kmap, dm, ws, cu, grid, st);
    case 5: return launch_g<5>(kmap, dm, ws, cu, grid, st);
    case 6: return launch_g<6>(kmap, dm, ws, cu, grid, st);
    case 7: return launch_g<7>(kmap, dm, ws, cu, grid, st);
    case 8: return launch_g<8>(kmap, dm, ws, cu, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace jacap
