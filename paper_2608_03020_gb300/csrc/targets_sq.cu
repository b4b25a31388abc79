// ||T_l||_F^2 of the feedback targets T_l = (E P_l) Q_l (S3, S11) without forming T_l:
//   ||T_l||^2 = sum_n u_n^T (Q_l Q_l^T) u_n,  u_n = e_n P_l
//             = < P_l (Q_l Q_l^T) P_l^T , E^T E >   (Frobenius inner product of two C x C matrices).
// The step of Eq. 10 needs it when the statistics kernel generates T itself (fused targets).
//
// k_tsq_ete    partial E^T E over chunks of TSQ_CHUNK tokens (products and sums in fp64), one C x C
//              slot per chunk.  Up to C = 16 the CTA's threads are split over entries and token
//              groups (summed in a fixed order): with one thread per entry, 16 threads walked
//              2048 tokens each (275 us at C = 4, N = 32768; 11 us now).
// k_tsq_block  a cluster of 8 CTAs per block l.  Each CTA forms M_l = Q_l Q_l^T over an eighth of the
//              channels (fp32 products over runs of at most 32 channels per lane, runs and lanes
//              summed in fp64, Q_l's slab staged in shared memory) and adds up the chunks' slots
//              of its share of the E^T E entries; CTA 0 reads both through distributed shared
//              memory in rank order and forms K = P_l M_l P_l^T and <K, E^T E> in fp64.
//              Latency-bound: one CTA per block took 63 us at L = 8, d = 3584, r = 16.
//              Deterministic.
#include <cooperative_groups.h>

#include "loca_internal.h"

namespace loca {
namespace {

constexpr int TSQ_THREADS = 256;
constexpr int TSQ_SPLIT = 8;      // CTAs per block in k_tsq_block
constexpr int TSQ_SLAB = 128;     // channels of Q staged at a time
constexpr int TSQ_CHUNK = 512;  // tokens per E^T E partial
constexpr int kMaxC = 64;
constexpr int kMaxR = 32;

__global__ void __launch_bounds__(TSQ_THREADS) k_tsq_ete(const float* __restrict__ E, int64_t N, int C,
                                                          double* __restrict__ part) {
  const int64_t n0 = int64_t(blockIdx.x) * TSQ_CHUNK;
  const int64_t n1 = n0 + TSQ_CHUNK < N ? n0 + TSQ_CHUNK : N;
  double* out = part + int64_t(blockIdx.x) * C * C;
  const int C2 = C * C;
  const int groups = C2 <= TSQ_THREADS ? TSQ_THREADS / C2 : 1;  // token groups per entry
  __shared__ double red[TSQ_THREADS];
  for (int e0 = 0; e0 < C2; e0 += TSQ_THREADS) {
    const int e = groups > 1 ? int(threadIdx.x) % C2 : e0 + int(threadIdx.x);
    const int grp = groups > 1 ? int(threadIdx.x) / C2 : 0;
    double acc = 0.0;
    if (e < C2 && grp < groups) {
      const int a = e / C, b = e % C;
#pragma unroll 8
      for (int64_t n = n0 + grp; n < n1; n += groups)
        if (LOCA_CHECK(n * C + a, N * C) && LOCA_CHECK(n * C + b, N * C)) acc = fma(double(E[n * C + a]), double(E[n * C + b]), acc);
    }
    if (groups > 1) {
      red[threadIdx.x] = acc;
      __syncthreads();
      if (threadIdx.x < C2)
        for (int q = 1; q < groups; ++q) acc += red[q * C2 + threadIdx.x];
    }
    if (grp == 0 && e < C2 && LOCA_CHECK(int64_t(blockIdx.x) * C2 + e, int64_t(gridDim.x) * C2)) out[e] = acc;
  }
}

__global__ void __cluster_dims__(TSQ_SPLIT, 1, 1) __launch_bounds__(TSQ_THREADS)
    k_tsq_block(const double* __restrict__ part, int nchunks, int C, const float* __restrict__ P,
                const float* __restrict__ Q, int r, int64_t d, double* __restrict__ tsq) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = int(cl.block_rank());
  constexpr int TT = TSQ_THREADS;
  __shared__ float Qs[kMaxR][TSQ_SLAB + 1];
  __shared__ double ete[kMaxC * kMaxC / TSQ_SPLIT];  // entries e with e % TSQ_SPLIT == rank
  __shared__ double M[kMaxR * (kMaxR + 1) / 2];      // upper triangle over this CTA's channels
  __shared__ double Mf[kMaxR * kMaxR];
  __shared__ double PM[kMaxC * kMaxR];
  __shared__ double red[TT];
  const int l = blockIdx.x / TSQ_SPLIT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int C2 = C * C;
  // E^T E entries of this CTA: one warp per entry, lanes over the chunks
  for (int e = rank + TSQ_SPLIT * warp; e < C2; e += TSQ_SPLIT * (TT / 32)) {
    double acc = 0.0;
    for (int c = lane; c < nchunks; c += 32) acc += part[int64_t(c) * C2 + e];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) ete[e / TSQ_SPLIT] = acc;
  }
  // M over this CTA's channels
  const float* Ql = Q + int64_t(l) * r * d;
  const int ntri = r * (r + 1) / 2;
  for (int e = threadIdx.x; e < ntri; e += TT) M[e] = 0.0;
  const int64_t per = (d + TSQ_SPLIT - 1) / TSQ_SPLIT;
  const int64_t cb = per * rank, ce = cb + per < d ? cb + per : d;
  for (int64_t c0 = cb; c0 < ce; c0 += TSQ_SLAB) {
    __syncthreads();
    for (int e = threadIdx.x; e < r * TSQ_SLAB; e += TT) {
      const int s = e / TSQ_SLAB, c = e % TSQ_SLAB;
      Qs[s][c] = (c0 + c < ce && LOCA_CHECK(int64_t(s) * d + c0 + c, int64_t(r) * d)) ? Ql[int64_t(s) * d + c0 + c] : 0.f;
    }
    __syncthreads();
    // one thread per entry: 4 runs of 32 channels
    for (int e = threadIdx.x; e < ntri; e += TT) {
      int si = 0, ti = e;  // e-th entry of the upper triangle
      while (ti >= r - si) ti -= r - si++;
      ti += si;
      double acc = 0.0;
#pragma unroll
      for (int c1 = 0; c1 < TSQ_SLAB; c1 += 32) {
        float run = 0.f;
#pragma unroll
        for (int c = 0; c < 32; ++c) run = fmaf(Qs[si][c1 + c], Qs[ti][c1 + c], run);
        acc += double(run);
      }
      M[e] += acc;
    }
  }
  cl.sync();
  if (rank == 0) {
    for (int e = threadIdx.x; e < ntri; e += TT) {
      double acc = 0.0;
      for (int q = 0; q < TSQ_SPLIT; ++q) acc += *cl.map_shared_rank(&M[e], q);
      int si = 0, ti = e;
      while (ti >= r - si) ti -= r - si++;
      ti += si;
      Mf[si * r + ti] = acc;
      Mf[ti * r + si] = acc;
    }
    __syncthreads();
    // PM = P_l M (C x r)
    const float* Pl = P + int64_t(l) * C * r;
    for (int e = threadIdx.x; e < C * r; e += TT) {
      const int a = e / r, t = e % r;
      double acc = 0.0;
      for (int s = 0; s < r; ++s) acc += double(Pl[a * r + s]) * Mf[s * r + t];
      PM[e] = acc;
    }
    __syncthreads();
    // <P M P^T, E^T E> = sum_ab (sum_t PM[a, t] P[b, t]) ete[a, b]
    double acc = 0.0;
    for (int e = threadIdx.x; e < C2; e += TT) {
      const int a = e / C, b = e % C;
      double k = 0.0;
      for (int t = 0; t < r; ++t) k += PM[a * r + t] * double(Pl[b * r + t]);
      acc += k * *cl.map_shared_rank(&ete[e / TSQ_SPLIT], e % TSQ_SPLIT);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0 && LOCA_CHECK(l, gridDim.x / TSQ_SPLIT)) {
      double t = 0.0;
      for (int w = 0; w < TT / 32; ++w) t += red[w];
      tsq[l] = t;
    }
  }
  cl.sync();  // no CTA leaves while CTA 0 may still read its partial sums
}

}  // namespace

int tsq_max_C() { return kMaxC; }
int tsq_max_r() { return kMaxR; }

size_t tsq_workspace_bytes(int64_t N, int C) {
  const int64_t nchunks = (N + TSQ_CHUNK - 1) / TSQ_CHUNK;
  return align256(sizeof(double) * size_t(nchunks > 0 ? nchunks : 1) * size_t(C) * size_t(C));
}

cudaError_t launch_targets_sq(const float* E, int64_t N, int C, const float* P, const float* Q, int L, int r,
                              int64_t d, double* tsq, void* workspace, cudaStream_t s) {
  const int64_t nchunks = (N + TSQ_CHUNK - 1) / TSQ_CHUNK;
  double* part = static_cast<double*>(workspace);
  if (nchunks > 0) k_tsq_ete<<<unsigned(nchunks), TSQ_THREADS, 0, s>>>(E, N, C, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_tsq_block<<<unsigned(L) * TSQ_SPLIT, TSQ_THREADS, 0, s>>>(part, int(nchunks), C, P, Q, r, d, tsq);
  return cudaGetLastError();
}

}  // namespace loca
