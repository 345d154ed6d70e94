// Orthogonalisation of an Arnoldi step: two classical Gram-Schmidt passes of
// the new vector w against the column's basis v_0..v_{nb-1}, its norm and the
// normalisation, in four launches over all iterating columns:
//
//   dots          d1_i = v_i . w
//   update, dots  w -= sum d1_i v_i, and at once d2_i = v_i . w
//   update, norm  w -= sum d2_i v_i, and at once w . w
//   scale         w *= 1 / ||w||
//
// A pass over the basis costs 4 nb + 1 FP64 multiply-adds per node (the FP64
// pipe issues one warp instruction per 16 cycles and SM: 0.6 T/s on the chip)
// and 3 nb + 7 vectors of traffic, which are near each other, so both the reads
// of the second pass's dots (taken from the update that just had the values in
// registers) and the reduction's additions count: a thread block's sums go
// through shared memory, 13 warp additions per dot, not 45 by shuffles.  No
// launch adds the partial sums up: each thread block of the next one does that
// for its column (nb sums of a few dozen values from L2).  The launches are
// chained by programmatic dependent launch.
//
// Measured against eight launches (dots, their sums and the update, twice; the
// norm, its sum, the scaling) that read the basis four times: the 21 steps of
// 64 columns of 180,000 nodes, bases of up to 7 vectors, 6.9 ms -> 4.5 ms
// (4.1 TB/s; 3.3 ms at the FP64 rate, 2.6 ms at the copy rate); 138 steps of
// 1 to 64 columns of 40,000 nodes 9.0 -> 4.7 ms; 27 steps of a few columns of
// 10,000 nodes, where the launches are all, 1.39 -> 0.56 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "kernels.h"

namespace matex {

namespace {

constexpr int kGsThreads = 256;
constexpr int kGsWarps = kGsThreads / 32;

struct GsArgs {
  double* Vb;
  int64_t vstride, n;
  const int32_t *slots, *iter;
  const double* in;  // partial sums of the previous launch, [K][nb][nch]
  double* out;       // those of this one
  SmallState ss;
  int chunk, nch, nb;
};

enum GsMode { kDots, kUpdateDots, kUpdateNorm };

__device__ __forceinline__ void gs_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ double gs_warp_sum(double v) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Total of partial sums p[0..nch), by one warp.  They and w are read past the L1
// cache: a launch of the chain may start while one two before it still reads
// the values they replace.
__device__ __forceinline__ double gs_total(const double* p, int nch) {
  double s = 0.0;
  for (int k = threadIdx.x & 31; k < nch; k += 32) s += __ldcg(p + k);
  return gs_warp_sum(s);
}

template <int NB, GsMode kMode>
__global__ void __launch_bounds__(kGsThreads) gs_pass_kernel(GsArgs a) {
  constexpr int kSums = kMode == kUpdateNorm ? 1 : NB;
  // nodes in flight per thread: two while their basis values fit the registers
  constexpr int U = NB <= 8 ? 2 : 1;
  __shared__ double red[kSums][kGsThreads];
  __shared__ double h[NB];
  const int warp = threadIdx.x >> 5;
  const int q = a.iter[blockIdx.y];
  double* __restrict__ base = a.Vb + (int64_t)a.slots[q] * a.vstride;
  double* __restrict__ w = base + (int64_t)NB * a.n;
  gs_wait();
  if (kMode != kDots) {
    double* __restrict__ col = a.ss.Ht + (int64_t)q * kMaxB * kMaxM + (NB - 1);
    for (int i = warp; i < NB; i += kGsWarps) {
      const double s = gs_total(a.in + ((int64_t)blockIdx.y * NB + i) * a.nch, a.nch);
      if ((threadIdx.x & 31) == 0) {
        h[i] = s;
        if (blockIdx.x == 0) col[i * kMaxM] += s;
      }
    }
    __syncthreads();
  }
  double acc[kSums];
#pragma unroll
  for (int i = 0; i < kSums; ++i) acc[i] = 0.0;
  const int64_t b = (int64_t)blockIdx.x * a.chunk;
  const int64_t e = min(a.n, b + a.chunk);
  for (int64_t x0 = b + threadIdx.x; x0 < e; x0 += U * kGsThreads) {
    double v[U][NB], wx[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t x = x0 + u * kGsThreads;
      const bool ok = x < e;
      wx[u] = ok ? __ldcg(w + x) : 0.0;
#pragma unroll
      for (int i = 0; i < NB; ++i) v[u][i] = ok ? base[(int64_t)i * a.n + x] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t x = x0 + u * kGsThreads;
      if (kMode != kDots) {
#pragma unroll
        for (int i = 0; i < NB; ++i) wx[u] = fma(-h[i], v[u][i], wx[u]);
        if (x < e) w[x] = wx[u];
      }
      if (kMode == kUpdateNorm) {
        if (x < e) acc[0] = fma(wx[u], wx[u], acc[0]);
      } else if (x < e) {
#pragma unroll
        for (int i = 0; i < kSums; ++i) acc[i] = fma(v[u][i], wx[u], acc[i]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kSums; ++i) red[i][threadIdx.x] = acc[i];
  __syncthreads();
  for (int i = warp; i < kSums; i += kGsWarps) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kGsWarps; ++k) s += red[i][32 * k + (threadIdx.x & 31)];
    s = gs_warp_sum(s);
    if ((threadIdx.x & 31) == 0)
      a.out[((int64_t)blockIdx.y * kSums + i) * a.nch + blockIdx.x] = s;
  }
}

__global__ void __launch_bounds__(kGsThreads) gs_scale_kernel(GsArgs a) {
  __shared__ double scale;
  const int q = a.iter[blockIdx.y];
  double* __restrict__ w = a.Vb + (int64_t)a.slots[q] * a.vstride + (int64_t)a.nb * a.n;
  gs_wait();
  if (threadIdx.x < 32) {
    const double nrm = sqrt(gs_total(a.in + (int64_t)blockIdx.y * a.nch, a.nch));
    if (threadIdx.x == 0) {
      scale = nrm > 0.0 ? 1.0 / nrm : 0.0;
      if (blockIdx.x == 0)
        a.ss.Ht[((int64_t)q * kMaxB + a.nb) * kMaxM + a.nb - 1] = nrm;
    }
  }
  __syncthreads();
  const double f = scale;
  const int64_t b = (int64_t)blockIdx.x * a.chunk;
  const int64_t e = min(a.n, b + a.chunk);
  for (int64_t x = b + threadIdx.x; x < e; x += kGsThreads) w[x] = __ldcg(w + x) * f;
}

// Nodes per thread block: 4096, so that the sums over a block (13 warp additions
// per dot against 128 multiply-adds) and over the blocks stay small, halved
// down to 512 while the launch has fewer than four blocks per SM.
constexpr int kGsChunk = 4096, kGsMinChunk = 512, kGsFill = 608;

int gs_chunk(int K, int64_t n) {
  int chunk = kGsChunk;
  while (chunk > kGsMinChunk && K * ((n + chunk - 1) / chunk) < kGsFill) chunk /= 2;
  return chunk;
}

template <typename Kernel>
void gs_launch(Kernel kernel, const GsArgs& a, int K, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)a.nch, (unsigned)K);
  cfg.blockDim = dim3(kGsThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, a);
}

template <int NB>
void gs_passes(GsArgs a, double* p0, double* p1, int K, cudaStream_t st) {
  a.out = p0;
  gs_launch(gs_pass_kernel<NB, kDots>, a, K, st);
  a.in = p0;
  a.out = p1;
  gs_launch(gs_pass_kernel<NB, kUpdateDots>, a, K, st);
  a.in = p1;
  a.out = p0;
  gs_launch(gs_pass_kernel<NB, kUpdateNorm>, a, K, st);
}

// partial sums of one launch: K columns of n nodes, at most kMaxM sums each
size_t gs_sums(int K, int64_t n) {
  const size_t full = (size_t)K * (size_t)((n + kGsChunk - 1) / kGsChunk);
  // a halved chunk was taken because twice its size gave fewer than kGsFill blocks
  return kMaxM * std::max(full, (size_t)2 * kGsFill);
}

}  // namespace

size_t gram_schmidt_partials(int K, int64_t n) { return 2 * gs_sums(K, n); }

int gram_schmidt(double* Vb, int64_t vstride, const int32_t* slots, const int32_t* iter, int K,
                 int nb, int64_t n, SmallState ss, double* partials, cudaStream_t st) {
  if (K <= 0 || nb < 1 || nb > kMaxM) return 0;
  GsArgs a = {Vb, vstride, n, slots, iter, nullptr, nullptr, ss, 0, 0, nb};
  a.chunk = gs_chunk(K, n);
  a.nch = (int)((n + a.chunk - 1) / a.chunk);
  double* p0 = partials;
  double* p1 = partials + gs_sums(K, n);
  switch (nb) {
#define MATEX_GS(NB) \
  case NB: gs_passes<NB>(a, p0, p1, K, st); break;
    MATEX_GS(1) MATEX_GS(2) MATEX_GS(3) MATEX_GS(4) MATEX_GS(5) MATEX_GS(6) MATEX_GS(7)
    MATEX_GS(8) MATEX_GS(9) MATEX_GS(10) MATEX_GS(11) MATEX_GS(12) MATEX_GS(13) MATEX_GS(14)
    MATEX_GS(15) MATEX_GS(16) MATEX_GS(17) MATEX_GS(18) MATEX_GS(19) MATEX_GS(20)
#undef MATEX_GS
  }
  a.in = p0;
  gs_launch(gs_scale_kernel, a, K, st);
  return 4;
}

}  // namespace matex
