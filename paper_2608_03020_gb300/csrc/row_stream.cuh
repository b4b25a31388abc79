// Streaming of token rows for the calibration kernels: a warp reads a piece of one row of a tall fp32
// matrix Y (tokens x w) per token, with a short vector V[token] (RP floats, the same for all lanes),
// and every lane works on its CPT columns of the row.
//
// Each warp has its own ring of two slots in shared memory, filled with cp.async (16 bytes a time, or 4
// when Y's rows are not 16-byte aligned) and drained without any barrier between warps, so a
// slot (4 KB of Y) is in flight while the other is used; sixteen warps an SM keep ~64 KB in flight,
// which the HBM latency needs and register-staged loads (16 KB at 160 registers a thread) did not
// reach.  The arithmetic is packed: fma.rn.f32x2 on pairs of V's entries.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "debug_check.cuh"

namespace loca {

__device__ __forceinline__ uint64_t f32x2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f32x2_parts(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {  // a - b
  return fma2(b, f32x2(-1.f, -1.f), a);  // exact product: one rounding
}

// Tokens per slot, and floats per slot: Y then V.
template <int RP, int CPT>
struct RowRing {
  static constexpr int TOK = CPT == 4 ? 8 : 16;
  static constexpr int COLS = 32 * CPT;
  static constexpr int Y_FLOATS = TOK * COLS;
  static constexpr int SLOT = Y_FLOATS + TOK * RP;
  static constexpr int BYTES = 2 * SLOT * 4;  // one warp's ring
};

__device__ __forceinline__ void cp_async(uint32_t dst, const float* src, int bytes, bool in) {
  const int n = in ? bytes : 0;  // bytes read; the rest of the destination is filled with zeros
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Start the copies of tokens [n0, n0 + TOK) (zeros from n1 on): columns [j0, j0 + COLS) of Y (zeros from
// w on) and V's rows, ldv floats apart.  vec: Y's rows and j0 are 16-byte aligned.  V and ldv always are.
template <int RP, int CPT>
__device__ __forceinline__ void row_issue(float* slot, const float* Y, int64_t w, int64_t j0, const float* V, int64_t ldv,
                                          int64_t n0, int64_t n1, bool vec, int lane) {
  using R = RowRing<RP, CPT>;
  const uint32_t sy = uint32_t(__cvta_generic_to_shared(slot));
  const uint32_t sv = sy + R::Y_FLOATS * 4;
  if (vec) {
    constexpr int PER = R::COLS / 4;  // 16-byte pieces per row
#pragma unroll
    for (int i = 0; i < R::TOK * PER / 32; ++i) {
      const int e = lane + 32 * i, t = e / PER, c = (e % PER) * 4;
      const bool in = n0 + t < n1 && j0 + c < w;
      cp_async(sy + uint32_t(t * R::COLS + c) * 4, in ? Y + (n0 + t) * w + j0 + c : Y, 16, in);
    }
  } else {
#pragma unroll 4
    for (int i = 0; i < R::TOK * R::COLS / 32; ++i) {
      const int e = lane + 32 * i, t = e / R::COLS, c = e % R::COLS;
      const bool in = n0 + t < n1 && j0 + c < w;
      cp_async(sy + uint32_t(e) * 4, in ? Y + (n0 + t) * w + j0 + c : Y, 4, in);
    }
  }
  constexpr int VP = RP / 4;
#pragma unroll
  for (int i = 0; i < (R::TOK * VP + 31) / 32; ++i) {
    const int e = lane + 32 * i, t = e / VP, c = (e % VP) * 4;
    if (e < R::TOK * VP) {
      const bool in = n0 + t < n1;
      cp_async(sv + uint32_t(e) * 16, in ? V + (n0 + t) * ldv + c : V, 16, in);
    }
  }
  cp_async_commit();
}

// A lane's CPT columns of token t of a slot, each duplicated into a pair.
template <int RP, int CPT>
__device__ __forceinline__ void row_cols(const float* slot, int t, int lane, float (&y)[CPT]) {
  const float* p = slot + t * RowRing<RP, CPT>::COLS + lane * CPT;
  if constexpr (CPT == 4) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    y[0] = v.x, y[1] = v.y, y[2] = v.z, y[3] = v.w;
  } else if constexpr (CPT == 2) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    y[0] = v.x, y[1] = v.y;
  } else {
    y[0] = *p;
  }
}

}  // namespace loca
