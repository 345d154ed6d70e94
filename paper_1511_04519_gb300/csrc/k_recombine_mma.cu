// Basis recombination on the tensor cores: the final step of
// Alg. 1 at every output of a segment round (Alg. 2's snapshots) and the sum of
// the groups' responses,
//   X[o][i] += sum over the round's columns q whose segment holds o of
//              V_q y_q(o) + (z_q - w_q) + (t_o - l_q) z'_q            (Eq. 6),
// as one contraction over k: a column's m basis vectors with the coefficients
// y_q(o), z'_q with t_o - l_q and z_q - w_q with 1, each zero where the column
// does not hold o.  Digit products of a 55-bit split (split8.cuh) on
// mma.sync: 16 outputs x 8 nodes over 16 terms take the FP64 pipe 1,024 clocks
// of an SM, the 34 digit products 68.
//
//   rm_list: the round's k in order of their columns' first outputs, so that
//     16 consecutive ones (a K step) live on few outputs, each with the power of
//     two that brings its vector to the size of its column's response: a
//     node's digits then start at the largest that any column has there, and an
//     output's at the columns' relative size at that time.  The error is below
//     2^-54 a term of the first times the second, so that small currents keep
//     their digits beside large ones and a long tail its own (currents of 1e-12
//     of the largest, at the nodes where they act: off by 2.5e-12 of the terms
//     with the bare vectors' digits, by less than 1e-13 with these);
//   rm_coef: per tile of 16 outputs the digits of the K steps that it meets,
//     and the set of those (a 64-bit mask);
//   rm_gemm: a CTA splits the vectors' values at its 32 nodes once, keeps the
//     digits (a byte each) in shared memory, and its eight warps walk the tiles
//     of outputs, one 8-node slice each, over the tiles' own K steps only: long
//     tails and short rise and fall segments alike do no work for padding
//     beyond their tiles.  X is read and written once per launch.
// Eight K steps make an exact sum (a chunk); rounds of more than 56 K steps take
// several launches.
//
// Measured on the 180k-node grid's tail round (64 columns, 237 basis vectors and
// 128 -P terms, 980 outputs, two thirds of the pairs held): 8.9 ms against 11.8 ms
// for nine 6-bit digits on tcgen05 with the -P terms in a pass of their own (one
// thread's issue of 990 M128 N48 products per 48 outputs, nine accumulators
// filling TMEM, and 72 KB of V digits re-read per 32 terms left its tensor pipe
// 4 % busy); the tensor pipe's own time is 5.6 ms.  Coefficients as bytes,
// widened by every warp: 10.1 ms.
#include <algorithm>

#include "kernels.h"
#include "split8.cuh"

namespace matex {

namespace {

using namespace s8;

constexpr int kRmThreads = 256;
constexpr int kRmNodes = 32;                      // nodes of a CTA
constexpr int kRmVStep = kRmNodes / 8 * kTileE;   // a K step's digits at those nodes
constexpr int kRmTile = kDigits * 512;            // coefficient tile, FP16 in fragment order
constexpr int kRmSmemMax = 224 * 1024;
constexpr int kRmMaxCh = kRmMaxSteps / kChunkSteps;

// One warp per column: exclusive sums over the columns in order, then the
// column's entries.  Entries past the total (only when a replay's counts
// disagree with the recording; the run is then discarded) are empty.
__global__ void __launch_bounds__(1024)
rm_list_kernel(RoundCols rc, const int32_t* __restrict__ order, const int32_t* __restrict__ mcol,
               const int32_t* __restrict__ tcut, const double* __restrict__ beta,
               const double* __restrict__ pbound, int K,
               int64_t vstride, int64_t gstride, int64_t n, RmK* __restrict__ list, int ktot, int kpad, unsigned long long* __restrict__ mask,
               int nmask) {
  __shared__ int warp_sum[32];
  __shared__ int base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < nmask; i += blockDim.x) mask[i] = 0;
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  for (int p0 = 0; p0 < K; p0 += blockDim.x) {
    const int p = p0 + (int)threadIdx.x;
    const int q = p < K ? (order ? order[p] : p) : 0;
    const int m = p < K ? mcol[q] : 0;
    int sum = p < K ? m + 2 : 0;
    const int cnt = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, sum, o);
      if (lane >= o) sum += v;
    }
    if (lane == 31) warp_sum[warp] = sum;
    __syncthreads();
    if (warp == 0) {
      int v = lane < (int)(blockDim.x >> 5) ? warp_sum[lane] : 0;
      const int own = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += x;
      }
      warp_sum[lane] = base + v - own;
      __syncwarp();
      if (lane == 31) base += v;
    }
    __syncthreads();
    if (p < K) {
      int k = warp_sum[warp] + sum - cnt;
      const int ob = rc.obeg[q], oe = ob + rc.nout[q];
      // tail skipping: past its cut a column loses V y, or all of it
      const int ov = tcut ? ob + tcut[2 * q] : oe;
      const int op = tcut && tcut[2 * q + 1] ? ov : oe;
      const int64_t vb = (int64_t)rc.vslot[q] * vstride, gb = (int64_t)rc.group[q] * gstride;
      auto size = [](double x) {  // its binary exponent, 0 for zero, inf and NaN
        const int e = (__double2hiint(x) >> 20) & 0x7ff;
        return e == 0 || e == 0x7ff ? 0 : e - 1022;
      };
      // the column's response: ||v|| V y, L z' and z - w; vectors of zeros stay out
      const double zw = pbound[2 * q], zp = pbound[2 * q + 1];
      const int sq = size(fmax(beta[q], fmax(zw, rc.len[q] * zp)));
      for (int j = 0; j < m && k < ktot; ++j, ++k) list[k] = RmK{vb + (int64_t)j * n, q, j, ob, ov, -sq, 0};
      if (k < ktot) list[k++] = RmK{zp == 0.0 ? -1 : gb, q, kMaxM, ob, op, size(zp) - sq, 0};
      if (k < ktot) list[k++] = RmK{zw == 0.0 ? -1 : gb, q, kMaxM + 1, ob, op, size(zw) - sq, 0};
    }
    __syncthreads();
  }
  for (int k = base + (int)threadIdx.x; k < kpad; k += blockDim.x) list[k] = RmK{-1, 0, 0, 0, 0, 0, 0};
}

// Coefficient tiles: blockIdx.x a tile of 16 outputs, blockIdx.y a chunk, warp
// w its K step.  Lane (g, t) holds outputs g, g + 8 and terms 2t, 2t + 1, 2t + 8,
// 2t + 9, mma.sync's A operand.
__global__ void __launch_bounds__(kRmThreads)
rm_coef_kernel(const RmK* __restrict__ list, int ksteps, const double* __restrict__ coef, int ldo,
               int obeg, int oend, unsigned char* __restrict__ tiles, int16_t* __restrict__ exps,
               unsigned long long* __restrict__ mask, const int32_t* __restrict__ abort) {
  if (abort && *abort) return;
  __shared__ int key[16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int ks = blockIdx.y * kChunkSteps + warp;
  const int o0 = obeg + blockIdx.x * 16;
  if (threadIdx.x < 16) key[threadIdx.x] = 0;
  __syncthreads();
  double v[2][4];
  bool any = false;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    RmK e{-1, 0, 0, 0, 0, 0, 0};
    if (ks < ksteps) e = list[ks * 16 + 2 * t + (u & 1) + (u >> 1) * 8];
    any |= e.off >= 0 && max(e.ob, o0) < min(e.oe, min(o0 + 16, oend));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int o = o0 + g + 8 * h;
      double x = 0.0;
      if (e.off >= 0 && o >= e.ob && o < e.oe && o < oend)
        x = ldexp(e.j > kMaxM ? 1.0 : coef[((int64_t)e.q * ldo + (o - e.ob)) * kCoefLd + e.j], e.sc);
      v[h][u] = x;
    }
  }
  const bool live = __any_sync(0xffffffffu, any);
  if (live) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int m = max(max(exp_key(v[h][0]), exp_key(v[h][1])), max(exp_key(v[h][2]), exp_key(v[h][3])));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
      if (t == 0) atomicMax(&key[g + 8 * h], m);
    }
    if (lane == 0) atomicOr(mask + blockIdx.x, 1ull << ks);
  }
  __syncthreads();
  if (threadIdx.x < 16)  // the chunk's exponents; 0x7fff: an inf or NaN among them
    exps[((size_t)blockIdx.x * gridDim.y + blockIdx.y) * 16 + threadIdx.x] =
        key[threadIdx.x] >= kKeyInf ? 0x7fff : (int16_t)key_exp(key[threadIdx.x]);
  if (!live) return;
  uint32_t lo[2][kDigits], hi[2][kDigits];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int e = key_exp(key[g + 8 * h]);
    widen_pair(digits(v[h][0], e), digits(v[h][1], e), lo[h]);
    widen_pair(digits(v[h][2], e), digits(v[h][3], e), hi[h]);
  }
  uint4* tile = reinterpret_cast<uint4*>(tiles + ((size_t)blockIdx.x * ksteps + ks) * kRmTile) + lane;
#pragma unroll
  for (int p = 0; p < kDigits; ++p) tile[32 * p] = make_uint4(lo[0][p], lo[1][p], hi[0][p], hi[1][p]);
}

struct RmArgs {
  double* Xp;
  int64_t n;
  const double *Vb, *Z, *Zp, *W;
  const RmK* list;
  const unsigned char* tiles;
  const int16_t* exps;
  const unsigned long long* mask;
  const double* coef;
  int ldo, ksteps, obeg, oend;
  const int32_t* abort;
};

// Chunk ch of output o at node i in FP64, the terms that hold o alone: taken
// where one of the chunk's values at i or of its coefficients at o is an inf or
// NaN, which has no digits and may belong to a column that does not hold o.
static __device__ __noinline__ double rm_plain(const RmArgs* a, int ch, int o, int64_t i) {
  const int k1 = min(a->ksteps, (ch + 1) * kChunkSteps) * 16;
  double s = 0.0;
  for (int k = ch * kChunkSteps * 16; k < k1; ++k) {
    const RmK e = a->list[k];
    if (e.off < 0 || o < e.ob || o >= e.oe) continue;
    const double v = e.j < kMaxM    ? a->Vb[e.off + i]
                     : e.j == kMaxM ? a->Zp[e.off + i]
                                    : a->Z[e.off + i] - a->W[e.off + i];
    s = fma(v, e.j > kMaxM ? 1.0 : a->coef[((int64_t)e.q * a->ldo + (o - e.ob)) * kCoefLd + e.j], s);
  }
  return s;
}

__global__ void __launch_bounds__(kRmThreads, 2) rm_gemm_kernel(const __grid_constant__ RmArgs a) {
  // [K step][8-node slice][digits 0..3 | 4, 5 | 6], then the CTA's tiles of
  // outputs (blockIdx.y, + gridDim.y, ...): their K steps and exponents
  extern __shared__ __align__(16) unsigned char rm_smem[];
  __shared__ int ek[kRmMaxCh][kRmNodes];
  if (a.abort && *a.abort) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int64_t i0 = (int64_t)blockIdx.x * kRmNodes;
  const int nch = (a.ksteps + kChunkSteps - 1) / kChunkSteps, ntile = (a.oend - a.obeg + 15) / 16;
  unsigned long long* mk = reinterpret_cast<unsigned long long*>(rm_smem + a.ksteps * kRmVStep);
  int16_t* eo = reinterpret_cast<int16_t*>(mk + ntile);
  for (int i = threadIdx.x; i < kRmMaxCh * kRmNodes; i += kRmThreads) (&ek[0][0])[i] = -kNonFinite;
  for (int i = threadIdx.x; i < ntile; i += kRmThreads) mk[i] = __ldg(a.mask + i);
  for (int i = threadIdx.x; i < ntile * nch * 8; i += kRmThreads)
    reinterpret_cast<int*>(eo)[i] = __ldg(reinterpret_cast<const int*>(a.exps) + i);
  __syncthreads();
  // ---- the vectors' digits at the CTA's nodes: warp items (K step, slice), lane
  // node g of the slice, terms 2t, 2t + 1, 2t + 8, 2t + 9 (mma.sync's B operand)
  const int items = a.ksteps * (kRmNodes / 8);
  auto load = [&](int it, double (&v)[4], int (&sc)[4]) {
    const int ks = it / (kRmNodes / 8);
    const int64_t i = i0 + (it % (kRmNodes / 8)) * 8 + g;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const RmK e = a.list[ks * 16 + 2 * t + (u & 1) + (u >> 1) * 8];
      double x = 0.0;
      if (e.off >= 0 && i < a.n)
        x = e.j < kMaxM ? a.Vb[e.off + i] : e.j == kMaxM ? a.Zp[e.off + i] : a.Z[e.off + i] - a.W[e.off + i];
      v[u] = x;
      sc[u] = e.sc;
    }
  };
  for (int it = warp; it < items; it += kRmThreads / 32) {
    double v[4];
    int sc[4], m = -kNonFinite;
    load(it, v, sc);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int key = exp_key(v[u]);
      m = max(m, key >= kKeyInf ? kNonFinite : key_exp(key) - sc[u]);
    }
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    if (t == 0)
      atomicMax(&ek[it / (kRmNodes / 8) / kChunkSteps][(it % (kRmNodes / 8)) * 8 + g], m);
  }
  __syncthreads();
  for (int it = warp; it < items; it += kRmThreads / 32) {
    double v[4];
    int sc[4];
    load(it, v, sc);
    const int e = ek[it / (kRmNodes / 8) / kChunkSteps][(it % (kRmNodes / 8)) * 8 + g];
    uint64_t d[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) d[u] = digits(v[u], e + sc[u]);
    uint32_t b[kDigits];
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
      const int sh = 8 * (6 - p);
      b[p] = (uint32_t)((d[0] >> sh) & 0xff) | (uint32_t)((d[1] >> sh) & 0xff) << 8 |
             (uint32_t)((d[2] >> sh) & 0xff) << 16 | (uint32_t)((d[3] >> sh) & 0xff) << 24;
    }
    unsigned char* s = rm_smem + it * kTileE;
    reinterpret_cast<uint4*>(s)[lane] = make_uint4(b[0], b[1], b[2], b[3]);
    reinterpret_cast<uint2*>(s + kTile45)[lane] = make_uint2(b[4], b[5]);
    reinterpret_cast<uint32_t*>(s + kTile6)[lane] = b[6];
  }
  __syncthreads();
  // ---- the tiles of outputs ----------------------------------------------------
  // A warp's (tile, K step) pairs in order.  The four warps of a tile read its
  // coefficients from L1 after the first; the next pair's digit d replaces the
  // current one's as soon as its last product is issued.  X of a tile is on its
  // way while the tensor core works.
  const int slice = warp & 3, stride = 2 * (int)gridDim.y;
  int fu = (warp >> 2) + 2 * (int)blockIdx.y - stride;
  unsigned long long fleft = 0;
  const uint4* fp = reinterpret_cast<const uint4*>(a.tiles) + lane;
  auto next = [&]() {
    while (!fleft) {
      fu += stride;
      if (fu >= ntile) return;
      fleft = mk[fu];
    }
    const int ks = __ffsll((long long)fleft) - 1;
    fleft &= fleft - 1;
    fp = reinterpret_cast<const uint4*>(a.tiles + ((size_t)fu * a.ksteps + ks) * kRmTile) + lane;
  };
  uint4 af[kDigits];
  next();
#pragma unroll
  for (int q = 0; q < kDigits; ++q) af[q] = __ldg(fp + 32 * q);
  for (int u = (warp >> 2) + 2 * (int)blockIdx.y; u < ntile; u += stride) {
    const unsigned long long m = mk[u];
    if (!m) continue;
    // outputs g (0, 1), g + 8 (2, 3) at nodes 2t, 2t + 1
    double xold[4], x[4];
    double* px = a.Xp + (int64_t)(a.obeg + u * 16 + g) * a.n + i0 + slice * 8 + 2 * t;
    auto live = [&](int i) {
      return a.obeg + u * 16 + g + 8 * (i >> 1) < a.oend && i0 + slice * 8 + 2 * t + (i & 1) < a.n;
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) xold[i] = live(i) ? px[(i >> 1) * 8 * a.n + (i & 1)] : 0.0;
    bool begun = false;
    for (int ch = 0; ch < nch; ++ch) {
      unsigned bits = (unsigned)(m >> (8 * ch)) & 0xffu;
      if (!bits) continue;
      const bool few = __popc(bits) <= 2;
      float c[4][kDigits];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < kDigits; ++q) c[i][q] = few || q < 2 ? kBiasedZero : 0.f;
      for (; bits; bits &= bits - 1) {
        const int ks = 8 * ch + __ffs((int)bits) - 1;
        next();  // past the last pair: the last one again
        const unsigned char* s = rm_smem + (ks * (kRmNodes / 8) + slice) * kTileE;
        const uint4 t0 = reinterpret_cast<const uint4*>(s)[lane];
        const uint2 t4 = reinterpret_cast<const uint2*>(s + kTile45)[lane];
        const uint32_t tp[kDigits] = {t0.x, t0.y, t0.z, t0.w, t4.x, t4.y,
                                      reinterpret_cast<const uint32_t*>(s + kTile6)[lane]};
#pragma unroll
        for (int p = 0; p < kDigits; ++p) {
          const uint32_t b0 = widen<0>(tp[p]), b1 = widen<1>(tp[p]);
#pragma unroll
          for (int r = 0; r + p < kDigits; ++r) mma(c, p + r, af[r], b0, b1);
          if (p > 0) {
            mma(c, kDigits - 1, af[kDigits - p], down8(b0), down8(b1));
            af[kDigits - p] = __ldg(fp + 32 * (kDigits - p));
          }
        }
        af[0] = __ldg(fp);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int en = ek[ch][slice * 8 + 2 * t + (i & 1)];  // a value's exponent, kNonFinite: an inf or NaN
        const int e = eo[(u * nch + ch) * 16 + g + 8 * (i >> 1)];
        double v = 0.0;
        if (en < kNonFinite && e != 0x7fff) {
          const int ee = e + en;
          v = few ? compose<true>(c[i], ee) : compose<false>(c[i], ee);
        } else if (live(i)) {
          v = rm_plain(&a, ch, a.obeg + u * 16 + g + 8 * (i >> 1), i0 + slice * 8 + 2 * t + (i & 1));
        }
        x[i] = begun ? x[i] + v : v;
      }
      begun = true;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (live(i)) px[(i >> 1) * 8 * a.n + (i & 1)] = xold[i] + x[i];
  }
}

}  // namespace

size_t rm_tiles_bytes(int n_times) { return (size_t)((n_times + 15) / 16) * kRmMaxSteps * kRmTile; }
size_t rm_exps(int n_times) { return (size_t)((n_times + 15) / 16) * kRmMaxCh * 16; }

bool rm_set_limits() {
  return cudaFuncSetAttribute(rm_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kRmSmemMax) == cudaSuccess;
}

int recombine_mma(double* Xp, int64_t n, const double* Vbase, int64_t vstride, const double* Z,
                  const double* Zp, const double* W, int64_t gstride, const RoundCols& rc,
                  const int32_t* order, const int32_t* mcol, const double* coef, int ldo, int K,
                  int kdim, int obeg_min, int oend_max, const RmScratch& rs, cudaStream_t st,
                  const double* beta, const double* pbound, const int32_t* tcut) {
  const int nt = (oend_max - obeg_min + 15) / 16;
  if (K <= 0 || nt <= 0) return 0;
  const int ktot = kdim + 2 * K, steps = (ktot + 15) / 16;
  // K steps of one launch: what fits shared memory beside its output tiles
  const int most = std::min(kRmMaxSteps, (kRmSmemMax - nt * (8 + 32 * kRmMaxCh)) / kRmVStep);
  const int parts = (steps + most - 1) / most;
  int launches = 1;
  rm_list_kernel<<<1, 1024, 0, st>>>(rc, order, mcol, tcut, beta, pbound, K, vstride, gstride, n, rs.list,
                                     ktot, steps * 16, rs.mask, nt * parts);
  for (int p = 0; p < parts; ++p) {
    const int s0 = steps * p / parts, ks = steps * (p + 1) / parts - s0;
    const RmK* list = rs.list + (size_t)s0 * 16;
    unsigned long long* mask = rs.mask + (size_t)p * nt;
    rm_coef_kernel<<<dim3((unsigned)nt, (unsigned)((ks + kChunkSteps - 1) / kChunkSteps)), kRmThreads, 0,
                     st>>>(list, ks, coef, ldo, obeg_min, oend_max, rs.tiles, rs.exps, mask, rc.abort);
    const unsigned gx = (unsigned)((n + kRmNodes - 1) / kRmNodes);
    // small grids: the tiles of outputs spread over more CTAs, about two per SM
    const unsigned gy = std::max(1u, std::min<unsigned>((unsigned)(nt + 1) / 2, 304u / gx));
    const int smem = ks * kRmVStep + nt * (8 + 32 * ((ks + kChunkSteps - 1) / kChunkSteps));
    rm_gemm_kernel<<<dim3(gx, gy), kRmThreads, smem, st>>>(
        RmArgs{Xp, n, Vbase, Z, Zp, W, list, rs.tiles, rs.exps, mask, coef, ldo, ks, obeg_min, oend_max, rc.abort});
    launches += 2;
  }
  return launches;
}

}  // namespace matex
