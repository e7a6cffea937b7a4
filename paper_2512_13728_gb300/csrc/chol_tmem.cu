// Cholesky factor and inverse of the first CholeskyQR pass for ranks up to 256 (tensor-core modes),
// with the working matrix in tensor memory.
//
// Same right-looking sweep as chol_inv_kernel (kernels_simt.cu) and chol_inv_tc_kernel (chol_tc.cu),
// over 32-wide block columns k (k0 = 32 k): before step k, rows i >= k0 of W hold the Schur
// complement in columns j >= k0 and U[i][j] = -sum_{K < k} L[i, K] L^{-1}[K, j] in columns j < k0.
// One CTA per layer.  W lives in TMEM: row i is lane i mod 128 of row block b = i / 128, its
// column j is TMEM column 128 b + j (block 0 needs 128 columns, block 1 256), so the rank-32 update
// W -= Yt Yt^T is a few MMAs that accumulate in place (A negated by the instruction descriptor),
// and W never crosses the memory system: S is read once and L^{-1} written once.  Warp w < 8 owns
// rows 32 w .. 32 w + 31.  Step k:
//   warp k      reads its 32 x 32 diagonal block and eliminates it, a helper warp of 8..15 carries
//               the inverse along (D_k = L_kk^{-1}, chol_blocks.cuh);
//   warps > k   read their rows of block column k (thread = row);
//   two helper warps of 8..15 whose TMEM lanes hold warp k's rows copy U[k, :k0] to shared memory;
//   -- barrier --
//   warps > k   form the panel L[i, k] = A[i, k] D_k^T;
//   warps < k   finish block row k: L^{-1}[k, q] = D_k U[k, q], thread = column q, and store it;
//   all eight   write their 32 rows of Yt (r x 32, K-major tf32 halves): L^{-1}[k, :k0 + 32]^T in
//               rows j < k0 + 32, the panel below;
//   -- barrier --
//   one thread  issues the update: first the 32 columns of block column k + 1, whose own barrier
//               lets the next step's factorization start under the rest.
// Rows above the block and columns right of the diagonal are dead: the MMAs write garbage there
// that nothing reads.  Block k's own columns start from zero (accumulate off) in the rows below.
// Bound by the serial diagonal blocks (chol_blocks.cuh).  The version that keeps W in global
// memory (TMA reduce-adds of drained TMEM tiles) took 98 us at r = 192 and 160 us at r = 256;
// this one 53 and 75 us (75 and 104 with the diagonal block in one warp).
// Accuracy: 3xTF32 (hi hi + hi lo + lo hi); any lower-triangular factor near L^{-1} serves here, as
// the second CholeskyQR pass measures and removes what it leaves.
#include "chol_blocks.cuh"
#include "common.cuh"
#include "tc.cuh"
#include "tc_common.cuh"

#include <algorithm>

namespace cd {
namespace {

using namespace tc;

constexpr int kThreads = 512;
constexpr int kUld = 260;  // row pitch of the U copy (16-byte writes of 8 consecutive rows: distinct banks)
constexpr int kDild = CB;  // row pitch of D_k
constexpr uint32_t kNegA = 1u << 13;  // instruction descriptor: A negated

// Rows of Yt: whole 128-row A operands.
__host__ __device__ constexpr int yt_rows(int r) { return r <= 128 ? 128 : 256; }

struct State {
  uint8_t *yth, *ytl;
  float *U, *DI;
  DiagScratch *diag;
  uint64_t *bars;  // [0]: block column k + 1 is updated; [1]: the whole update is done; [2]: drain
  uint32_t tmem;
  uint32_t it;     // updates issued so far in this kernel
  int *bad, *gave_up;
};

__device__ __forceinline__ uint32_t w_col(uint32_t tmem, int b, int j) { return tmem + 128u * b + j; }

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]), "f"(v[16]), "f"(v[17]), "f"(v[18]),
      "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]), "f"(v[24]), "f"(v[25]), "f"(v[26]), "f"(v[27]),
      "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_ldf(uint32_t taddr, float (&v)[32]) {
  uint32_t u[32];
  tmem_ld32(taddr, u);
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(u[i]);
}

// Row `row` of Yt as its hi and lo tf32 halves, in the 128-byte-swizzled layout.
__device__ __forceinline__ void write_yt(const State &st, int row, const float (&v)[CB]) {
#pragma unroll
  for (int c4 = 0; c4 < 8; ++c4) {
    float h[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float x = v[4 * c4 + e];
      h[e] = __uint_as_float(__float_as_uint(x) & 0xFFFFE000u);
      lo[e] = x - h[e];
    }
    const uint32_t off = sw128_f32((uint32_t)row, (uint32_t)c4);
    *reinterpret_cast<float4 *>(st.yth + off) = make_float4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<float4 *>(st.ytl + off) = make_float4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// W[block b][n0 .. n0 + nn) -= Yt[block b] Yt[n0 ..]^T, starting from zero when `fresh`.
__device__ __forceinline__ void issue(const State &st, int b, int n0, int nn, bool fresh) {
  const uint32_t ah = smem_u32(st.yth) + (uint32_t)b * 16384u, al = smem_u32(st.ytl) + (uint32_t)b * 16384u;
  const uint32_t bh = smem_u32(st.yth) + (uint32_t)n0 * 128u, bl = smem_u32(st.ytl) + (uint32_t)n0 * 128u;
  const uint32_t idesc = idesc_tf32(128, (uint32_t)nn, false, false) | kNegA, d = w_col(st.tmem, b, n0);
  uint64_t dah = smem_desc_sw128(ah, 0, 1024), dal = smem_desc_sw128(al, 0, 1024);
  uint64_t dbh = smem_desc_sw128(bh, 0, 1024), dbl = smem_desc_sw128(bl, 0, 1024);
#pragma unroll
  for (int k8 = 0; k8 < 4; ++k8, dah += 2, dal += 2, dbh += 2, dbl += 2) {  // 32 bytes, in units of 16
    umma_tf32(d, dah, dbl, idesc, fresh && k8 == 0 ? 0u : 1u);
    umma_tf32(d, dal, dbh, idesc, 1u);
    umma_tf32(d, dah, dbh, idesc, 1u);
  }
}

// 0: factored; 1: a pivot was not positive and finite (uniform over the block); 2: a wait for the
// tensor cores gave up.
__device__ int sweep(const float *S, const float *S2, float *__restrict__ W, int r, int64_t ls, float shift, State &st,
                     int32_t *status) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rw = warp & 7, row = 32 * rw + lane;  // the rows whose TMEM lanes this warp can reach
  const uint32_t lanes = (uint32_t)(32 * (warp & 3)) << 16;
  const int nblk = (r + CB - 1) / CB;
  // W <- lower triangle of S (+ S2) + shift I; zeros past r.  Warps rw and rw + 8 share the 32-column
  // chunks of rows 32 rw ..; the columns right of the diagonal chunk are never read.
  for (int c = warp >> 3; c <= rw && rw < yt_rows(r) / 32; c += 2) {
    float v[32];
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      const int j = 32 * c + 4 * g;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
      if (row < r && j < r) {  // pitch: a multiple of 8
        x = *reinterpret_cast<const float4 *>(S + (int64_t)row * ls + j);
        if (S2 != nullptr) y = *reinterpret_cast<const float4 *>(S2 + (int64_t)row * ls + j);
      }
      v[4 * g] = x.x + y.x; v[4 * g + 1] = x.y + y.y; v[4 * g + 2] = x.z + y.z; v[4 * g + 3] = x.w + y.w;
    }
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      if (32 * c + e >= r) v[e] = 0.f;
      if (32 * c + e == row && row < r) v[e] += shift;
    }
    tmem_st32(w_col(st.tmem, rw >> 2, 32 * c) + lanes, v);
  }
  tmem_st_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  for (int k = 0; k < nblk; ++k) {
    const int k0 = CB * k, nb = min(CB, r - k0), R0 = k0 + nb;
    const uint32_t par = (st.it - 1u) & 1u;  // the previous step's update (k > 0)
    float v[CB];
    if (warp < 8) {
      if (warp >= k && warp < nblk) {
        if (k > 0 && !mbar_wait(&st.bars[0], par, status)) *st.gave_up = 1;
        tc_fence_after();
        tmem_ldf(w_col(st.tmem, warp >> 2, k0) + lanes, v);
      }
      if (warp == k) {  // lane i holds row k0 + i (identity padding below a short block)
#pragma unroll
        for (int j = 0; j < CB; ++j) {
          if (j > lane || lane >= nb) v[j] = 0.f;
          if (j == lane && lane >= nb) v[j] = 1.f;
        }
        const bool ok = diag_factor<1>(v, *st.diag, lane);
        if (lane == 0) *st.bad = ok ? 0 : 1;
      }
    } else if ((warp & 3) == (k & 3)) {
      // the whole update of the previous step is done: U[k, :k0] is final and Yt may be rewritten
      if (k > 0 && !mbar_wait(&st.bars[1], par, status)) *st.gave_up = 1;
      tc_fence_after();
      for (int c = (warp >> 2) & 1; c < k; c += 2) {
        tmem_ldf(w_col(st.tmem, k >> 2, 32 * c) + lanes, v);
#pragma unroll
        for (int g = 0; g < 8; ++g)
          *reinterpret_cast<float4 *>(st.U + lane * kUld + 32 * c + 4 * g) =
              make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
      }
    } else {
      const int h = ((warp >> 2) & 1) * 3 + (((warp & 3) - (k & 3) - 1) & 3);  // 0 .. 5
      if (h == 0) {  // D_k = L_kk^{-1}, a segment of columns behind warp k
        diag_invert<1, kDild>(*st.diag, st.DI, lane);
      } else {  // zeros right of the diagonal block in block row k of L^{-1}
        for (int i = h - 1; i < nb; i += 5)
          for (int c = R0 + lane; c < r; c += 32) W[(int64_t)(k0 + i) * ls + c] = 0.f;
      }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (*st.gave_up) return 2;
    if (*st.bad) return 1;
    if (warp < nblk) {
      if (warp == k) {  // rows k0 .. k0 + 31 of Yt: the columns of D_k
#pragma unroll
        for (int c = 0; c < CB; ++c) v[c] = st.DI[c * kDild + lane];
      } else {
        if (warp < k) {  // column q = row: the finished L^{-1}[k, q] = D_k U[k, q]
#pragma unroll
          for (int c = 0; c < CB; ++c) v[c] = st.U[c * kUld + row];
        }
        trmv32<CB - 1, kDild>(v, st.DI);  // or the panel row L[row, k] = A[row, k] D_k^T
      }
      if (warp <= k) {
#pragma unroll
        for (int c = 0; c < CB; ++c)
          if (c < nb && row < r) W[(int64_t)(k0 + c) * ls + row] = v[c];
      }
      if (R0 < r) write_yt(st, row, v);
    }
    if (R0 >= r) break;
    fence_async_smem();  // the Yt writes are read by the tensor cores
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == kThreads - 32) {
      // columns R0 .. (the next block column) first, then the others
      const int np = (r + 15) / 16 * 16, first = min(CB, np - R0);
      for (int b = 0; b < 2; ++b)
        if (R0 < 128 * (b + 1) && 128 * b < r) issue(st, b, R0, first, false);
      umma_commit(&st.bars[0]);
      for (int b = 0; b < 2; ++b) {
        if (R0 >= 128 * (b + 1) || 128 * b >= r) continue;
        const int n1 = min(np, 128 * (b + 1));
        if (k0 > 0) issue(st, b, 0, k0, false);
        issue(st, b, k0, CB, true);
        if (R0 + CB < n1) issue(st, b, R0 + CB, n1 - R0 - CB, false);
      }
      umma_commit(&st.bars[1]);
    }
    ++st.it;
  }
  return 0;
}

__global__ void __launch_bounds__(kThreads, 1) chol_inv_tmem_kernel(Shared sh) {
  chain_enter();
  const int l = blockIdx.x;
  if (!sh.active[l]) return;
  const DevLayer &Ly = sh.layers[l];
  const int r = (int)Ly.r;
  if (r > kCholTmemRank) return;  // chol_inv_tc_kernel's
  const int64_t ls = Ly.ldp;
  const float *S = Ly.S;
  float *Li = Ly.Linv;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = align1024(smem_raw);
  __shared__ uint32_t tmem_base_s;
  __shared__ int bad, gave_up;
  __shared__ double red[kThreads / 32];
  __shared__ double trace_s;
  __shared__ uint64_t bars_s[3];
  const int ya = yt_rows(r), tid = threadIdx.x;
  State st;
  st.yth = smem;
  st.ytl = smem + (size_t)ya * 128;
  st.U = reinterpret_cast<float *>(st.ytl + (size_t)ya * 128);  // CB x kUld
  st.DI = st.U + CB * kUld;                                     // CB x kDild
  st.diag = reinterpret_cast<DiagScratch *>(st.DI + CB * kDild);
  st.bars = bars_s;
  st.it = 0;
  st.bad = &bad;
  st.gave_up = &gave_up;
  const uint32_t cols = r <= 128 ? 128u : 512u;
  // two partial sums are added on their way into TMEM; more, in a pass of their own (its coalesced
  // reads keep more in flight: eight parts at r = 192 cost 8 us, added on the way 20)
  const float *S2 = Ly.s_parts == 2 ? S + Ly.s_stride : nullptr;
  if (Ly.s_parts > 2) sum_gram_parts<kThreads>(Ly.S, r, ls, Ly.s_parts, Ly.s_stride);
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) mbar_init(&bars_s[i], 1);
    gave_up = 0;
    fence_mbar_init();
  }
  if ((tid >> 5) == 0) {
    tmem_alloc(&tmem_base_s, cols);
    tmem_relinquish();
  }
  // rows of Yt past the last block stay zero
  for (int e = tid; e < ya * 8; e += kThreads) {
    reinterpret_cast<float4 *>(st.yth)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    reinterpret_cast<float4 *>(st.ytl)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  st.tmem = tmem_base_s;

  int res;
  bool shifted = false;
  float shift = 0.f;
#pragma unroll 1
  for (;;) {
    res = sweep(S, S2, Li, r, ls, shift, st, sh.status);
    if (res != 1 || shifted) break;
    // a retry from S + s I (shifted CholeskyQR, as in chol_inv_kernel)
    double tr = 0.0;
    for (int i = tid; i < r; i += kThreads)
      tr += (double)S[(int64_t)i * ls + i] + (S2 != nullptr ? (double)S2[(int64_t)i * ls + i] : 0.0);
    tr = block_sum<kThreads>(tr, red);
    if (tid == 0) trace_s = tr;
    __syncthreads();
    const double u = 5.9604644775390625e-8;  // 2^-24
    shift = (float)(11.0 * ((double)Ly.m * r + (double)r * (r + 1)) * u * trace_s);
    shifted = true;
    if (!(trace_s > 0.0 && isfinite(trace_s))) break;
  }
  if (tid == 0) {
    sh.orth_shifted[l] = shifted ? 1 : 0;
    if (shifted) atomicAdd(&sh.gate_scratch[kScratchShifted], 1ull);
  }
  if (res != 0) {
    if (tid == kThreads - 32) {
      if (res == 1) set_status(sh.status, ST_BREAKDOWN);
      umma_commit(&bars_s[2]);  // every MMA issued so far has completed before TMEM is freed
      mbar_wait(&bars_s[2], 0, sh.status);
    }
    __syncthreads();
    for (int64_t e = tid; e < (int64_t)r * r; e += kThreads) Li[(e / r) * ls + e % r] = 0.f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if ((tid >> 5) == 0) tmem_dealloc(st.tmem, cols);
}

}  // namespace

cudaError_t prepare_chol_inv_tmem(size_t *smem_out) {
  *smem_out = 1024 + 2 * (size_t)yt_rows(kCholTmemRank) * 128 + sizeof(float) * (CB * kUld + CB * kDild) + sizeof(DiagScratch);
  return allow_dynamic_smem(chol_inv_tmem_kernel, *smem_out);
}

void launch_chol_inv_tmem(const Shared &sh, size_t smem, cudaStream_t s) {
  if (sh.num_layers > 0) launch_chained(chol_inv_tmem_kernel, sh.num_layers, kThreads, smem, s, sh);
}

}  // namespace cd
