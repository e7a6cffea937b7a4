// Error feedback + parameter update (Algorithm 1/2, sync branch):
//   M = B - (1 - mu) P R^T,   X = X - eta sqrt(m/n) P Q_t^T
// run as one persistent, warp-specialized kernel over 256 x 128 output tiles, one CTA pair per
// tile (CTA c owns its rows 128 c .. 128 c + 127):
//   warp 0      TMA producer: bf16 K-major chunks of P (A: this CTA's 128 rows) and of R and Q_t
//               (B: this CTA's half, 64 of the tile's 128 rows) into a shared-memory ring
//               (BF16X3: also their low halves);
//   warp 1      (CTA 0) MMA issuer: two 256x128x16 pair MMAs per k-step into a double-buffered
//               pair of TMEM accumulators (U1 = P R^T, U2 = P Q_t^T; 4 x 128 = 512 columns);
//   warp 6      streams: TMA loads of 128 x 32 boxes of M, X (and G) into a ring of sub-chunk
//               buffers, TMA stores of the buffers the epilogue has finished;
//   warps 2..5  epilogue (thread = tile row): U1/U2 from TMEM, M_t and X_t computed in place in the
//               sub-chunk buffers; per-tile fp64 partial of ||M_t||^2 for Equation 1.
// HBM-bound.  The streams have a warp of their own, so that no epilogue thread waits for a store to
// be read before the next load goes out, and move 128-byte row segments (64-byte ones reached 6.0
// TB/s at rank 48, these 6.3); the pair MMA halves the R and Q_t bytes each SM receives, which pays
// for the larger stream buffers.  Measured before (a CTA per 128 x 128 tile, 64-byte segments issued
// by the epilogue's first thread, a barrier per sub-chunk), with a stream warp alone, and now:
// 290 / 262 / 250 us on the 160M stack at rank 192, 542 / 475 / 455 us on half of the 350M stack
// (B in M), 1003 / 917 / 829 us on all of it with split operands, 3826 / 4075 / 3650 us on the 1.3B
// stack at rank 512.  The same loads as cp.async copies from four more warps: 257, 459, 943, 4024.
#include "tc.cuh"
#include "tc_common.cuh"
#include "tc_kernels.cuh"

#include <algorithm>

namespace cd {
namespace tc {

// ============================================================ update (tcgen05) kernel ===
constexpr int U_SUB = 32;                        // columns of a stream sub-chunk: 128-byte row segments
constexpr uint32_t U_EBOX = 128u * U_SUB * 4u;  // one 128 x 32 fp32 box of M or X (128-byte swizzle)
constexpr uint32_t U_GBOX = 128u * U_SUB * 2u;  // one 128 x 32 bf16 box of G (64-byte swizzle)
constexpr int U_THREADS = 7 * 32;
constexpr uint32_t U_IDESC = idesc_bf16(256, 128, false, false);
// Ring depths.  A stage holds this CTA's 128 rows of P and its 64 rows of R and of Q_t: BF16 in
// 64-wide K chunks (128-byte swizzle); BF16X3, with the low halves too (P R^T = Ph Rh^T + Ph Rl^T
// + Pl Rh^T, the same for P Q_t^T), in 32-wide K chunks (64-byte swizzle): 32 KB either way.  The
// rest of shared memory holds stream sub-chunks of M, X and, where the kernel forms B = M + G
// itself (GIN), G: 40 KB or 32 KB each.
// DEEP takes a fourth operand stage and a stream buffer less, for ranks above kDeepRank: there a
// tile's operands (r / 64 chunks of 32 KB) outweigh its streams, and more stream loads in flight
// only delay them.  DEEP / not, us: forming B itself (GIN) 459 / 484 on twelve 1024-wide blocks at
// rank 256, 255 / 250 on the 160M stack at rank 192; with B in M 977 / 1058 on twelve 1536-wide
// blocks at rank 384, 461 / 468 on eight 1280-wide ones at rank 320, 440 / 410 at rank 256.  Four
// stream buffers with B in M: 484 us for 455 with three on half of the 350M stack.  BF16X3 fits four
// stages and three buffers: 829 us on the 350M stack, 905 with three stages.
constexpr int kDeepRankG = 224, kDeepRank = 288;  // with G; with B in M (between the ranks measured on either side)
template <bool X3, bool GIN, bool DEEP>
struct UpdCfg {
  static constexpr uint32_t KW = X3 ? 32u : 64u;  // K chunk width (bf16 elements per operand row)
  static constexpr uint32_t PB = 128u * KW * 2u, BB = 64u * KW * 2u;  // bytes of a P box, of an R or Q_t box
  static constexpr uint32_t HALF = PB + 2u * BB;  // P, R, Q_t; BF16X3: then their low halves
  static constexpr int STAGES = DEEP || X3 ? 4 : 3;
  static constexpr uint32_t STAGE = (X3 ? 2u : 1u) * HALF;
  static constexpr int EBUF = DEEP ? 2 : 3;
  static constexpr uint32_t EBUFB = 2u * U_EBOX + (GIN ? U_GBOX : 0u);  // bytes of one sub-chunk buffer
  static constexpr uint32_t SMEM = 1024u + STAGES * STAGE + EBUF * EBUFB + 256u;
  static_assert(EBUFB % 1024u == 0 && HALF % 1024u == 0, "every box stays aligned to its swizzle atom");
  static_assert(SMEM <= 227u * 1024u, "update smem");
  static_assert((2 * STAGES + 4 + 2 * EBUF + 1) * 8 <= 256, "barriers");
};

// Tile = {layer, row-tile pair p, column tile, ||M_t|| slot of row tile 2 p}.
template <bool X3, bool GIN, bool DEEP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(U_THREADS, 1)
    tc_update_kernel(Shared sh, const int4 *__restrict__ tiles, const int *__restrict__ off, const LayerMaps *__restrict__ maps,
                     float mu, float eta, float keep) {
  chain_enter();
  using Cfg = UpdCfg<X3, GIN, DEEP>;
  constexpr int U_STAGES = Cfg::STAGES, U_EBUF = Cfg::EBUF;
  constexpr uint32_t U_STAGE = Cfg::STAGE, U_EBUFB = Cfg::EBUFB;
  constexpr uint32_t KW = Cfg::KW, PB = Cfg::PB, BB = Cfg::BB, HALF = Cfg::HALF;
  if (sh.gate_scratch[kScratchActive] == 0ull) return;  // no layer takes the Dion branch
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = align1024(smem_raw);
  uint8_t *stage = smem;
  uint8_t *epi = smem + U_STAGES * U_STAGE;
  uint64_t *bars = reinterpret_cast<uint64_t *>(epi + U_EBUF * U_EBUFB);
  uint64_t *full = bars, *empty = bars + U_STAGES;
  uint64_t *acc_full = bars + 2 * U_STAGES, *acc_empty = acc_full + 2, *epi_full = acc_empty + 2;
  uint64_t *epi_done = epi_full + U_EBUF, *drain = epi_done + U_EBUF;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  __shared__ double red_s[4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // hand-off waits between the roles use the plan's limit; the drains below keep the default
  const Abort ab{&abort_s, sh.handoff_limit_ns};
  const uint32_t rank = cluster_ctarank();  // row tile 2 p + rank of the segment's tiles
  const int seg = blockIdx.x >> 1;
  // 32-column sub-chunks of a tile that start inside the matrix; 0 for the pair's second tile
  // when it lies past the last row tile
  auto subs_of = [&](const int4 &t) -> int {
    const DevLayer &L = sh.layers[t.x];
    if ((int64_t)(2 * t.y + (int)rank) * 128 >= L.m) return 0;
    return (int)min((int64_t)(128 / U_SUB), (L.n - (int64_t)t.z * 128 + U_SUB - 1) / U_SUB);
  };

  if (threadIdx.x == 0) {
    for (int i = 0; i < U_STAGES; ++i) {
      mbar_init(&full[i], 1);   // used in CTA 0: its arm, both CTAs' bytes
      mbar_init(&empty[i], 1);  // pair commit after the stage's MMAs
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);   // pair commit after the tile's MMAs
      mbar_init(&acc_empty[b], 2);  // used in CTA 0: each CTA's epilogue leader, its warps having read TMEM
    }
    for (int b = 0; b < U_EBUF; ++b) {
      mbar_init(&epi_full[b], 1);  // the sub-chunk's loads
      mbar_init(&epi_done[b], 4);  // one arrival per epilogue warp: M_t and X_t are in the buffer
    }
    mbar_init(drain, 1);
    abort_s = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(&tmem_base_s, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_sync();  // both CTAs' barriers and TMEM exist before anything crosses the pair
  const uint32_t tmem = tmem_base_s;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int ti = off[seg]; ti < off[seg + 1] && ok; ++ti) {
        const int4 t = tiles[ti];
        if (!sh.active[t.x]) continue;
        const LayerMaps *mp = maps + t.x;
        const int kch = (int)((sh.layers[t.x].r + KW - 1) / KW);
        const int mb = 2 * t.y + (int)rank;  // past the last row tile: zero-filled, not stored
        for (int kc = 0; kc < kch; ++kc, ++it) {
          const uint32_t s = it % U_STAGES, ph = (it / U_STAGES) & 1u;
          if (!ab.wait(&empty[s], ph ^ 1u, sh.status)) { ok = false; break; }
          uint8_t *sp = stage + s * U_STAGE;
          const uint32_t fb = cluster_addr(&full[s], 0);
          if (rank == 0) mbar_expect_tx(&full[s], 2u * U_STAGE);
          const int k0 = kc * (int)KW, b0 = t.z * 128 + (int)rank * 64;
          if (X3) {
            tma_load_2d_pair(sp, &mp->P_hi32, fb, k0, mb * 128);
            tma_load_2d_pair(sp + PB, &mp->R_hi32, fb, k0, b0);
            tma_load_2d_pair(sp + PB + BB, &mp->Qn_hi32, fb, k0, b0);
            tma_load_2d_pair(sp + HALF, &mp->P_lo32, fb, k0, mb * 128);
            tma_load_2d_pair(sp + HALF + PB, &mp->R_lo32, fb, k0, b0);
            tma_load_2d_pair(sp + HALF + PB + BB, &mp->Qn_lo32, fb, k0, b0);
          } else {
            tma_load_2d_pair(sp, &mp->P_hi, fb, k0, mb * 128);
            tma_load_2d_pair(sp + PB, &mp->R_64, fb, k0, b0);
            tma_load_2d_pair(sp + PB + BB, &mp->Qn_mn, fb, k0, b0);
          }
        }
      }
      // drain: the last stages' loads have landed and been consumed (their stage was freed); after
      // an abort the first wait that runs out has given every load far longer than it takes
      for (uint32_t k = (it > U_STAGES ? it - U_STAGES : 0); k < it; ++k)
        if (!mbar_wait(&empty[k % U_STAGES], (k / U_STAGES) & 1u, sh.status)) break;
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0 && rank == 0) {
      uint32_t it = 0, tcount = 0;
      bool ok = true;
      const uint64_t sd0 = X3 ? smem_desc_sw64(smem_u32(stage), 512) : smem_desc_sw128(smem_u32(stage), 0, 1024);
      for (int ti = off[seg]; ti < off[seg + 1] && ok; ++ti) {
        const int4 t = tiles[ti];
        if (!sh.active[t.x]) continue;
        const int kch = (int)((sh.layers[t.x].r + KW - 1) / KW);
        const uint32_t b = tcount & 1u, aph = (tcount >> 1) & 1u;
        if (!ab.wait<true>(&acc_empty[b], aph ^ 1u, sh.status)) break;
        tc_fence_after();
        const uint32_t d1 = tmem + b * 256u, d2 = d1 + 128u;
        for (int kc = 0; kc < kch; ++kc, ++it) {
          const uint32_t s = it % U_STAGES, ph = (it / U_STAGES) & 1u;
          if (!ab.wait(&full[s], ph, sh.status)) { ok = false; break; }
          tc_fence_after();
          const uint64_t sd = desc_at(sd0, s * U_STAGE);
          // K-major operand box at offset o of the stage, advanced by k16 steps of 16 elements (32 bytes)
          auto desc = [&](uint32_t o, int k16) { return desc_at(sd, o + (uint32_t)k16 * 32u); };
#pragma unroll
          for (int k16 = 0; k16 < (int)(KW / 16u); ++k16) {
            const uint64_t ad = desc(0, k16), rd = desc(PB, k16), qd = desc(PB + BB, k16);
            const uint32_t acc = (kc | k16) ? 1u : 0u;
            umma_pair_bf16(d1, ad, rd, U_IDESC, acc);
            umma_pair_bf16(d2, ad, qd, U_IDESC, acc);
            if (X3) {  // P R^T = Ph Rh^T + Ph Rl^T + Pl Rh^T, P Q_t^T likewise
              const uint64_t adl = desc(HALF, k16);
              umma_pair_bf16(d1, ad, desc(HALF + PB, k16), U_IDESC, 1u);
              umma_pair_bf16(d1, adl, rd, U_IDESC, 1u);
              umma_pair_bf16(d2, ad, desc(HALF + PB + BB, k16), U_IDESC, 1u);
              umma_pair_bf16(d2, adl, qd, U_IDESC, 1u);
            }
          }
          umma_pair_commit_mc(&empty[s], 0x3);  // the stage is free in both CTAs once its MMAs have read it
        }
        if (!ok) break;
        umma_pair_commit_mc(&acc_full[b], 0x3);
        ++tcount;
      }
      umma_pair_commit(drain);  // every MMA of the pair has completed before TMEM is freed
      mbar_wait(drain, 0, sh.status);
    }
  } else if (warp == 6) {
    // ---------------------------------------------------------------- streams of M, X and G
    // Loads run as far ahead of the epilogue as there are buffers, across tile boundaries (they do
    // not depend on the MMAs): the next load into a buffer goes out as soon as its store has been
    // read.
    if (lane == 0) {
      const int tend = off[seg + 1];
      int lt = off[seg], lj = 0;  // load cursor: tile, sub-chunk
      auto skip_empty = [&]() {
        while (lt < tend && (!sh.active[tiles[lt].x] || subs_of(tiles[lt]) == 0)) ++lt;
      };
      skip_empty();
      uint32_t issued = 0, stored = 0;
      auto load_next = [&]() {  // the next sub-chunk, into the buffer of sub-chunk issued - U_EBUF
        const int4 t = tiles[lt];
        const LayerMaps *mp = maps + t.x;
        const uint32_t eb = issued % U_EBUF;
        uint8_t *bs = epi + eb * U_EBUFB;
        const int r0 = (2 * t.y + (int)rank) * 128, x0 = t.z * 128 + lj * U_SUB;
        const bool defer = GIN && sh.layers[t.x].b_deferred != 0;  // B = M + G is formed here
        mbar_expect_tx(&epi_full[eb], 2u * U_EBOX + (defer ? U_GBOX : 0u));
        tma_load_2d(bs, &mp->Mf, &epi_full[eb], x0, r0);
        tma_load_2d(bs + U_EBOX, &mp->Xf, &epi_full[eb], x0, r0);
        if (defer) tma_load_2d(bs + 2 * U_EBOX, &mp->Gh32, &epi_full[eb], x0, r0);
        ++issued;
        if (++lj == subs_of(t)) {
          lj = 0;
          ++lt;
          skip_empty();
        }
      };
      while (issued < (uint32_t)U_EBUF && lt < tend) load_next();
      bool ok = true;
      for (int ti = off[seg]; ti < tend && ok; ++ti) {
        const int4 t = tiles[ti];
        if (!sh.active[t.x]) continue;
        const LayerMaps *mp = maps + t.x;
        const int ns = subs_of(t), r0 = (2 * t.y + (int)rank) * 128;
        for (int sub = 0; sub < ns; ++sub, ++stored) {
          const uint32_t eb = stored % U_EBUF;
          if (!ab.wait(&epi_done[eb], (stored / U_EBUF) & 1u, sh.status)) { ok = false; break; }
          uint8_t *bs = epi + eb * U_EBUFB;
          const int x0 = t.z * 128 + sub * U_SUB;  // past the matrix's edges: clipped by the store
          tma_store_2d(&mp->Mf, bs, x0, r0);
          tma_store_2d(&mp->Xf, bs + U_EBOX, x0, r0);
          bulk_commit();
          if (lt < tend) {
            bulk_wait_read<0>();
            load_next();
          }
        }
      }
      bulk_wait<0>();
      // every load has landed (after an abort the epilogue may not have waited for the last ones):
      // the latest load of each buffer, whose phase is the barrier's latest
      for (uint32_t k = issued > (uint32_t)U_EBUF ? issued - U_EBUF : 0u; k < issued; ++k)
        mbar_wait(&epi_full[k % U_EBUF], (k / U_EBUF) & 1u, sh.status);
    }
  } else {
    // ---------------------------------------------------------------- epilogue (128 threads)
    const int et = threadIdx.x - 64;
    const uint32_t row = 32u * (warp & 3) + lane;  // TMEM lane = tile row
    const bool leader = (et == 0);
    const int tend = off[seg + 1];
    uint32_t tcount = 0, ecount = 0;
    for (int ti = off[seg]; ti < tend; ++ti) {
      const int4 t = tiles[ti];
      if (!sh.active[t.x]) continue;
      const DevLayer &L = sh.layers[t.x];
      const float dec = 1.f - mu, c = eta * L.sqrt_m_over_n;
      const int ntc = (int)((L.n + 127) / 128);
      const int ns = subs_of(t);
      const bool defer = GIN && L.b_deferred != 0;
      const uint32_t b = tcount & 1u, aph = (tcount >> 1) & 1u;
      if (!named_and(1, 128, ab.wait(&acc_full[b], aph, sh.status))) break;
      tc_fence_after();
      float ss = 0.f;
      bool ok = true;  // warp-uniform; the four warps agree at the tile's last barrier
      for (int j = 0; j < ns; ++j) {  // sub-chunk j = 32-column TMEM chunk j
        uint32_t u1[32], u2[32];
        tmem_ld32(tmem + ((32u * (warp & 3)) << 16) + b * 256u + j * 32, u1);
        tmem_ld32(tmem + ((32u * (warp & 3)) << 16) + b * 256u + 128u + j * 32, u2);
        tmem_ld_wait();
        const uint32_t k = ecount + j, eb = k % U_EBUF, eph = (k / U_EBUF) & 1u;
        if (!__all_sync(0xffffffffu, ab.wait(&epi_full[eb], eph, sh.status))) {
          ok = false;
          break;
        }
        uint8_t *bs = epi + eb * U_EBUFB;
#pragma unroll
        for (int q = 0; q < U_SUB / 4; ++q) {
          const uint32_t o = sw128_f32(row, q);
          float4 bv = *reinterpret_cast<float4 *>(bs + o);
          float4 xv = *reinterpret_cast<float4 *>(bs + U_EBOX + o);
          if (defer) {  // B = M_{t-1} + G, the same fp32 additions as the buffer pass
            const uint2 gv =
                *reinterpret_cast<const uint2 *>(bs + 2 * U_EBOX + sw64_f32(row, (uint32_t)q >> 1) + (q & 1) * 8);
            bv.x += __uint_as_float(gv.x << 16);
            bv.y += __uint_as_float(gv.x & 0xffff0000u);
            bv.z += __uint_as_float(gv.y << 16);
            bv.w += __uint_as_float(gv.y & 0xffff0000u);
          }
          bv.x = fmaf(-dec, __uint_as_float(u1[4 * q + 0]), bv.x);
          bv.y = fmaf(-dec, __uint_as_float(u1[4 * q + 1]), bv.y);
          bv.z = fmaf(-dec, __uint_as_float(u1[4 * q + 2]), bv.z);
          bv.w = fmaf(-dec, __uint_as_float(u1[4 * q + 3]), bv.w);
          xv.x = fmaf(-c, __uint_as_float(u2[4 * q + 0]), xv.x * keep);  // keep: decoupled weight decay
          xv.y = fmaf(-c, __uint_as_float(u2[4 * q + 1]), xv.y * keep);
          xv.z = fmaf(-c, __uint_as_float(u2[4 * q + 2]), xv.z * keep);
          xv.w = fmaf(-c, __uint_as_float(u2[4 * q + 3]), xv.w * keep);
          ss = fmaf(bv.x, bv.x, ss); ss = fmaf(bv.y, bv.y, ss);
          ss = fmaf(bv.z, bv.z, ss); ss = fmaf(bv.w, bv.w, ss);
          *reinterpret_cast<float4 *>(bs + o) = bv;
          *reinterpret_cast<float4 *>(bs + U_EBOX + o) = xv;
        }
        fence_async_smem();  // the buffer is read by the stream warp's store
        __syncwarp();
        if (lane == 0) mbar_arrive(&epi_done[eb]);
      }
      ecount += ns;
      // per-tile ||M_t||^2 (rows/columns outside the matrix hold 0), fixed reduction order;
      // the barrier also ends every thread's TMEM reads of this accumulator
      const float ss1[1] = {ss};
      const double v = warp_sum_pairs<1>(ss1);
      if (lane == 0) red_s[warp - 2] = v;
      tc_fence_before();
      if (!named_and(1, 128, ok)) break;
      if (leader) {
        mbar_arrive_cluster(cluster_addr(&acc_empty[b], 0));  // every thread has read accumulator buffer b
        if (ns > 0) sh.upart[t.w + (int)rank * ntc] = (red_s[0] + red_s[1]) + (red_s[2] + red_s[3]);
      }
      ++tcount;
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs are done with the pair's TMEM and barriers
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, 512);
}

// ========================================================================= launch ===
template <bool X3, bool GIN, bool DEEP>
cudaError_t setup() {
  return allow_dynamic_smem(tc_update_kernel<X3, GIN, DEEP>, UpdCfg<X3, GIN, DEEP>::SMEM);
}
cudaError_t setup_update_kernel(bool x3) {
  if (x3) return setup<true, false, false>();
  for (const cudaError_t e : {setup<false, true, false>(), setup<false, false, false>(), setup<false, true, true>(),
                              setup<false, false, true>()})
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

template <bool X3, bool GIN, bool DEEP>
static void launch_as(const Shared &sh, const TcPlan &tp, float mu, float eta, float keep, cudaStream_t s) {
  launch_chained(tc_update_kernel<X3, GIN, DEEP>, 2 * tp.d_update.grid, U_THREADS, UpdCfg<X3, GIN, DEEP>::SMEM, s, 
      sh, tp.d_update.tiles, tp.d_update.off, tp.maps, mu, eta, keep);
}

void launch_update(const Shared &sh, const TcPlan &tp, float mu, float eta, float keep, cudaStream_t s) {
  if (tp.d_update.grid <= 0) return;
  const bool gin = tp.defers && !sh.b_in_m;  // else B is in M
  const bool deep = tp.max_r > (gin ? kDeepRankG : kDeepRank);
  if (tp.precision == DION_PREC_BF16X3) launch_as<true, false, false>(sh, tp, mu, eta, keep, s);
  else if (gin && deep) launch_as<false, true, true>(sh, tp, mu, eta, keep, s);
  else if (gin) launch_as<false, true, false>(sh, tp, mu, eta, keep, s);
  else if (deep) launch_as<false, false, true>(sh, tp, mu, eta, keep, s);
  else launch_as<false, false, false>(sh, tp, mu, eta, keep, s);
}

}  // namespace tc
}  // namespace cd
