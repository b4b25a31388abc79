// Small positive-definite solves shared by the ridge-solve kernels (S7: no explicit inverse).
//
// The k x k system matrix (k <= KM) lives in shared memory in fp64; the whole block factors it
// (Cholesky, right-looking, one barrier per column); every thread then solves its own right-hand
// side rows by a forward and a back substitution in fp32 registers.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace loca {

// Factor Md = L L^T (lower triangle of the leading k x k part; overwritten) with every thread of the
// block, filling Lf (KM x KM fp32 lower factor, rows 16-byte aligned; identity beyond k) and Linv (fp32
// reciprocals of its diagonal).  Returns 0, or c + 1 when the leading minor of order c + 1 is not
// positive definite.  Bound by the latency of its k steps (a reciprocal square root and two barriers
// each) and the fp64 pipe, 2 operations per clock and SM: the trailing entries of a step are dealt
// out one by one, two rows of the triangle folded into one of constant length.
template <int KM>
__device__ int chol_factor(double (*Md)[KM], float (*Lf)[KM], float* Linv, int k) {
  __shared__ double col[KM];
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int e = tid; e < KM * KM; e += nt) Lf[e / KM][e % KM] = (e / KM == e % KM) ? 1.f : 0.f;
  for (int a = tid; a < KM; a += nt) Linv[a] = 1.f;
  __syncthreads();
  for (int c = 0; c < k; ++c) {
    const double piv = Md[c][c];
    if (!(piv > 0.0)) return c + 1;  // the same value in every thread
    const double inv = rsqrt(piv);
    for (int a = c + 1 + tid; a < k; a += nt) {
      const double v = Md[a][c] * inv;
      col[a] = v;
      Lf[a][c] = float(v);
    }
    if (tid == 0) {
      Lf[c][c] = float(piv * inv);
      Linv[c] = float(inv);
    }
    __syncthreads();
    // rows c + 1 + i, i < rem, with i + 1 entries each: rows i and rem - 1 - i side by side
    const int rem = k - 1 - c, width = rem + 1;
    const uint32_t magic = (65536u + uint32_t(width) - 1u) / uint32_t(width);  // e / width for e width < 2^16
    for (int e = tid; e < (rem + 1) / 2 * width; e += nt) {
      int i = int((uint32_t(e) * magic) >> 16), j = e - i * width;
      if (j > i) {
        if (rem - 1 - i == i) continue;  // the middle row stands alone
        j -= i + 1;
        i = rem - 1 - i;
      }
      Md[c + 1 + i][c + 1 + j] = fma(-col[c + 1 + i], col[c + 1 + j], Md[c + 1 + i][c + 1 + j]);
    }
    __syncthreads();
  }
  return 0;
}

// c[i] <- c[i] (L L^T)^-1 for NR rows (length KM) in registers.  Both substitutions read the rows of L, four
// entries at a time: forward as dot products, backward by removing a solved entry from the earlier
// ones.  Bound by the shared loads, hence several rows per thread.  The warp barriers keep the compiler
// from holding the factor in registers from one pass to the other (2 KB of spills a thread at KM = 32).
template <int KM, int NR>
__device__ __forceinline__ void chol_solve_rows(const float (*Lf)[KM], const float* Linv, float (*c)[KM]) {
#pragma unroll
  for (int s = 0; s < KM; ++s) {
    if (KM >= 16) __syncwarp();
#pragma unroll
    for (int t = 0; t < s; t += 4) {
      const float4 v = *reinterpret_cast<const float4*>(&Lf[s][t]);
      const float l4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + u < s)
#pragma unroll
          for (int i = 0; i < NR; ++i) c[i][s] = fmaf(-l4[u], c[i][t + u], c[i][s]);
    }
    const float di = Linv[s];
#pragma unroll
    for (int i = 0; i < NR; ++i) c[i][s] *= di;
  }
#pragma unroll
  for (int s = KM - 1; s >= 0; --s) {
    if (KM >= 16) __syncwarp();
    const float di = Linv[s];
#pragma unroll
    for (int i = 0; i < NR; ++i) c[i][s] *= di;
#pragma unroll
    for (int t = 0; t < s; t += 4) {
      const float4 v = *reinterpret_cast<const float4*>(&Lf[s][t]);
      const float l4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (t + u < s)
#pragma unroll
          for (int i = 0; i < NR; ++i) c[i][t + u] = fmaf(-l4[u], c[i][s], c[i][t + u]);
    }
  }
}

// c[i] += b M for row-major M (rows of KM floats, 16-byte aligned shared memory), one row t of M and one
// entry b[i] = bt[i] of each of the NR rows.
template <int KM, int NR>
__device__ __forceinline__ void add_scaled_row(const float* row, const float (&bt)[NR], float (*c)[KM]) {
#pragma unroll
  for (int s = 0; s < KM; s += 4) {
    const float4 v = *reinterpret_cast<const float4*>(row + s);
    const float m4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int i = 0; i < NR; ++i) c[i][s + u] = fmaf(bt[i], m4[u], c[i][s + u]);
  }
}

// Rows of k floats to and from registers (16-byte accesses where the rows allow them).
template <int KM>
__device__ __forceinline__ void store_row(float* dst, const float* c, int k, bool vec) {
  if (vec) {
#pragma unroll
    for (int s = 0; s < KM; s += 4)
      if (s < k) *reinterpret_cast<float4*>(dst + s) = make_float4(c[s], c[s + 1], c[s + 2], c[s + 3]);
  } else {
#pragma unroll
    for (int s = 0; s < KM; ++s)
      if (s < k) dst[s] = c[s];
  }
}
template <int KM>
__device__ __forceinline__ void add_row(const float* src, float* c, int k, bool vec) {
  if (vec) {
#pragma unroll
    for (int s = 0; s < KM; s += 4)
      if (s < k) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(src + s));
        c[s] += v.x, c[s + 1] += v.y, c[s + 2] += v.z, c[s + 3] += v.w;
      }
  } else {
#pragma unroll
    for (int s = 0; s < KM; ++s)
      if (s < k) c[s] += __ldg(src + s);
  }
}

// Rows per thread of the row solves where there are plenty: register room for NR x KM sums.  Problems
// of fewer rows than the chip has threads take one.
__host__ __device__ constexpr int chol_rows_per_thread(int km) { return km <= 8 ? 4 : 2; }

}  // namespace loca
