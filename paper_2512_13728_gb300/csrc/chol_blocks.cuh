// 32 x 32 diagonal-block building blocks of the Cholesky + L^{-1} kernels (kernels_simt.cu:
// FFMA sweep; chol_tmem.cu and chol_tc.cu: sweeps with the trailing update on tensor cores).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace cd {

constexpr int CB = 32;

// Row-tile index of tile p in a lower trapezoid whose row tile b holds c1 + b tiles: the
// largest b with b c1 + b (b - 1) / 2 <= p.
// fp32 estimate (p < 2^21 here), corrected exactly in integers.
__device__ __forceinline__ int trap_row(int p, int c1) {
  const float bq = 2.f * (float)c1 - 1.f;
  int b = (int)((sqrtf(bq * bq + 8.f * (float)p) - bq) * 0.5f);
  if (b < 0) b = 0;
  while ((b + 1) * c1 + (b + 1) * b / 2 <= p) ++b;
  while (b > 0 && b * c1 + b * (b - 1) / 2 > p) --b;
  return b;
}

__device__ __forceinline__ void load8(const float *p, float w[8]) {
  const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
  w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
}
__device__ __forceinline__ void store8(float *p, const float w[8]) {
  *reinterpret_cast<float4 *>(p) = make_float4(w[0], w[1], w[2], w[3]);
  *reinterpret_cast<float4 *>(p + 4) = make_float4(w[4], w[5], w[6], w[7]);
}

// Unrolled through template recursion so that every register array is indexed by constants (no
// local-memory copies).
// v <- T v for a lower-triangular 32 x 32 T (row-major, row pitch LD), in place from the bottom.
template <int C, int LD = CB>
__device__ __forceinline__ void trmv32(float (&v)[CB], const float *T) {
  if constexpr (C >= 0) {
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int c2 = 0; c2 <= C; c2 += 2) {
      a0 = fmaf(T[C * LD + c2], v[c2], a0);
      if (c2 + 1 <= C) a1 = fmaf(T[C * LD + c2 + 1], v[c2 + 1], a1);
    }
    v[C] = a0 + a1;
    trmv32<C - 1, LD>(v, T);
  }
}

// Cholesky factor and inverse of a 32 x 32 block by two warps.  The first (diag_factor) eliminates
// the columns, lane = row; the second (diag_invert) carries the inverse along one eight-column
// segment behind, lane = column.  Both are loops over the columns of a segment, in registers that
// move down one place per column (v[0] is the current column), so that the code stays small (fully
// unrolled columns cost 20K cycles of instruction fetches the first time through) and the work
// shrinks with the segments.  Bound by the elimination's chain from column to column; about 5K
// cycles against 12.6K for one warp that factored with unrolled shuffles and then inverted.
struct alignas(16) DiagScratch {
  // current column, unscaled, from the pivot down; [CB]: the next diagonal entry ([CB + 1]: dump for
  // the lanes that do not hold it, which spares the loop a divergent branch)
  float col[2][CB + 4];
  float t[CB][CB];  // t[J][i - J] = a_iJ / pivot_J below the pivot, else 0
  float rs[CB];     // 1 / sqrt(pivot_J)
};
template <int ID>
__device__ __forceinline__ void diag_arrive() { asm volatile("bar.arrive %0, 64;" ::"n"(ID) : "memory"); }
template <int ID>
__device__ __forceinline__ void diag_sync() { asm volatile("bar.sync %0, 64;" ::"n"(ID) : "memory"); }

struct DiagState {
  float piv, rs, next;  // this column's pivot, its reciprocal square root, the next diagonal entry
  float4 a;             // the column's first four entries from the pivot down
};
__device__ __forceinline__ void diag_column(DiagScratch &sc, DiagState &ds, int J, int lane, float v0, float v1) {
  float *col = sc.col[J & 1];
  col[(lane - J) & 31] = lane >= J ? v0 : 0.f;
  col[lane == J + 1 ? CB : CB + 1] = v1;
  __syncwarp();
  ds.a = *reinterpret_cast<const float4 *>(col);
  ds.next = col[CB];
}
// Columns 32 - N .. 39 - N: v[0 .. N) hold this lane's row from column 32 - N on.  Every lane also
// works out the next pivot (the lane that holds it does not use its own), and the next column is on its
// way through shared memory before this one's multiply-adds, which run under both latencies.
template <int N>
__device__ __forceinline__ void diag_factor_segment(float (&v)[CB], DiagState &ds, DiagScratch &sc, int lane) {
#pragma unroll 1
  for (int J = CB - N; J < CB - N + 8; ++J) {
    const float *col = sc.col[J & 1];
    const float4 a = ds.a;
    // scaled twice by 1 / sqrt(pivot): 1 / pivot itself overflows for a subnormal pivot
    const float t = lane > J ? (v[0] * ds.rs) * ds.rs : 0.f, l1 = a.y * ds.rs;
    const float v0 = fmaf(-t, a.y, v[1]), v1 = fmaf(-t, a.z, v[2]), v2 = fmaf(-t, a.w, v[3]);
    sc.rs[J] = ds.rs;
    ds.piv = fmaf(-l1, l1, ds.next);
    ds.rs = rsqrtf(ds.piv);
    diag_column(sc, ds, J + 1, lane, v0, v1);
    sc.t[J][(lane - J) & 31] = t;
    v[0] = v0;
    v[1] = v1;
    v[2] = v2;
#pragma unroll
    for (int q = 1; q < N / 4; ++q) {
      const float4 b = *reinterpret_cast<const float4 *>(col + 4 * q);
      v[4 * q - 1] = fmaf(-t, b.x, v[4 * q]);
      v[4 * q] = fmaf(-t, b.y, v[4 * q + 1]);
      v[4 * q + 1] = fmaf(-t, b.z, v[4 * q + 2]);
      v[4 * q + 2] = fmaf(-t, b.w, v[4 * q + 3]);
    }
    __syncwarp();  // every lane has read this column: the next iteration writes its buffer
  }
}
// v: this lane's row of the block (entries right of the diagonal are not used).  Returns whether
// every pivot was positive and finite.  ID .. ID + 3: named barriers shared with diag_invert.
template <int ID>
__device__ __forceinline__ bool diag_factor(float (&v)[CB], DiagScratch &sc, int lane) {
  DiagState ds;
  ds.piv = __shfl_sync(0xffffffffu, v[0], 0);
  ds.rs = rsqrtf(ds.piv);
  diag_column(sc, ds, 0, lane, v[0], v[1]);
  diag_factor_segment<32>(v, ds, sc, lane);
  diag_arrive<ID>();
  diag_factor_segment<24>(v, ds, sc, lane);
  diag_arrive<ID + 1>();
  diag_factor_segment<16>(v, ds, sc, lane);
  diag_arrive<ID + 2>();
  diag_factor_segment<8>(v, ds, sc, lane);
  diag_arrive<ID + 3>();
  __syncwarp();
  const float mine = sc.rs[lane];  // a pivot that is not positive and finite leaves NaN, inf or 0
  return __all_sync(0xffffffffu, mine > 0.f && mine < INFINITY);
}

// Rows 32 - N .. 39 - N of the inverse: x[0 .. N) hold this lane's column from row 32 - N on.
template <int N, int LD>
__device__ __forceinline__ void diag_invert_segment(float (&x)[CB], const DiagScratch &sc, float *DI, int lane) {
#pragma unroll 1
  for (int J = CB - N; J < CB - N + 8; ++J) {
    const float cur = x[0];
    DI[J * LD + lane] = cur * sc.rs[J];
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
      const float4 b = *reinterpret_cast<const float4 *>(sc.t[J] + 4 * q);
      if (q > 0) x[4 * q - 1] = fmaf(-b.x, cur, x[4 * q]);
      x[4 * q] = fmaf(-b.y, cur, x[4 * q + 1]);
      x[4 * q + 1] = fmaf(-b.z, cur, x[4 * q + 2]);
      x[4 * q + 2] = fmaf(-b.w, cur, x[4 * q + 3]);
    }
  }
}
// DI <- the inverse of the factor, row-major with row pitch LD.
template <int ID, int LD>
__device__ __forceinline__ void diag_invert(const DiagScratch &sc, float *DI, int lane) {
  float x[CB];
#pragma unroll
  for (int c = 0; c < CB; ++c) x[c] = (c == lane) ? 1.f : 0.f;
  diag_sync<ID>();
  diag_invert_segment<32, LD>(x, sc, DI, lane);
  diag_sync<ID + 1>();
  diag_invert_segment<24, LD>(x, sc, DI, lane);
  diag_sync<ID + 2>();
  diag_invert_segment<16, LD>(x, sc, DI, lane);
  diag_sync<ID + 3>();
  diag_invert_segment<8, LD>(x, sc, DI, lane);
}

// Row i and 16-byte column group j4 (4 j4 <= i) of flat group p of a lower triangle whose rows
// 4 b .. 4 b + 3 hold b + 1 groups each, 2 b (b + 1) groups before them (p < 2^24: the fp32
// estimate of b is off by at most one, corrected in integers; 32-bit division).
__device__ __forceinline__ void lower_group(int64_t p, int &i, int &j4) {
  const uint32_t pu = (uint32_t)p;
  uint32_t b = (uint32_t)((sqrtf(2.f * (float)pu + 1.f) - 1.f) * 0.5f);
  while (2u * (b + 1u) * (b + 2u) <= pu) ++b;
  while (b > 0u && 2u * b * (b + 1u) > pu) --b;
  const uint32_t off = pu - 2u * b * (b + 1u), q = off / (b + 1u);
  i = (int)(4u * b + q);
  j4 = (int)(off - q * (b + 1u));
}

// S (lower triangle) += its other `parts` - 1 partial sums, `stride` floats apart, in order, by a
// block of THREADS threads; visible to the whole block on return.
template <int THREADS>
__device__ __forceinline__ void sum_gram_parts(float *S, int r, int64_t ls, int parts, int64_t stride) {
  if (parts <= 1) return;
  const int nb4 = r / 4, groups = 2 * nb4 * (nb4 + 1) + (r % 4) * (nb4 + 1);
  constexpr int U = 4;  // groups in flight per thread and part
  for (int g0 = threadIdx.x; g0 < groups; g0 += THREADS * U) {
    float4 a[U];
    float *p[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      int i = 0, j4 = 0;
      if (g0 + u * THREADS < groups) lower_group(g0 + u * THREADS, i, j4);
      p[u] = S + (int64_t)i * ls + 4 * j4;
      a[u] = *reinterpret_cast<const float4 *>(p[u]);
    }
#pragma unroll 2
    for (int q = 1; q < parts; ++q) {
      float4 b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) b[u] = *reinterpret_cast<const float4 *>(p[u] + q * stride);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        a[u].x += b[u].x; a[u].y += b[u].y; a[u].z += b[u].z; a[u].w += b[u].w;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (g0 + u * THREADS < groups) *reinterpret_cast<float4 *>(p[u]) = a[u];
  }
  __syncthreads();
}

}  // namespace cd
