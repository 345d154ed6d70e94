// Multi-right-hand-side level solves on the tensor cores: every supernode's
// product of the substitutions (the operator apply of Alg. 1 and the input
// solves of Eq. 5/6),
//   forward : [y_s; u_R] = P_s b_s, then b_R -= u_R (FP64 atomics),
//   backward: x_s = P_s^T [D_s^{-1} y_s; -x_R],
// as FP16 digit products (34 per tile), as accurate as FP64 relative to the
// largest entries of a panel row and of a right-hand side over 128 terms
// (split8.cuh).  The FP64 pipe (two FMA per clock and SM on GB300) bounds
// k_sptrsv.cu: 8 panel rows x 16 right-hand sides over 16 terms take it 1,024
// clocks of an SM, the 34 digit products of the same tile take mma.sync 68
// (measured: 2.0 clocks each).  mma.sync rather than tcgen05 because panels
// are small and ragged (on the 180k-node grid 48 x 95 on average): a warp
// works on 8 x 16 panel tiles in registers, with no TMEM or 128-row tile to
// fill.
//
// One launch per tree level and direction, chained by programmatic dependent
// launch.  A CTA takes either a pack of small supernodes or a block of row
// tiles of a larger one, for 16 right-hand sides:
//   1. its slice of the right-hand sides is split once: warps take fragments
//      of 16 terms, the largest exponent of a column meets in shared memory,
//      and the FP16 digits land there in fragment order;
//   2. each warp takes row tiles: 34 mma.sync per K step, the right-hand sides
//      as A operand, the panel as B (8 rows: little padding), its digits (one
//      byte each, split once at setup, with the signs of -u_R and -x_R and
//      with D^{-1}) from a ring of tiles that the warp fills by cp.async: a
//      load takes 1,500 clocks and more, a K step 290 and more.  The ring's
//      first tiles are under way before the previous level completes;
//   3. the seven integer sums become one FP64 value.
// A reduction longer than 128 terms runs in chunks whose FP64 values are
// added; where a level has few tasks, a thread-block cluster shares the
// chunks of a task, each CTA writing its values into the shared memory of the
// one that adds them up, in rank order.
//
// Two sizes of CTA.  Four warps, four CTAs an SM, one warp per row tile, where
// the level fills the GPU: there the tensor pipe and the issue slots count.
// Eight warps where every CTA of the level is resident at once: the level then
// lasts as long as one CTA does, and two warps per row tile, each with half of
// its K steps and of the right-hand sides' splitting, shorten that (13,000
// clocks to 9,000 from the previous level's end on: 1,900 until it is seen,
// 1,700 for the right-hand sides, 800 to split them, 2,500 for up to four K
// steps of two warps per scheduler, 600 for the conversion, 1,000 to 2,500 for
// the sums).
//
// Measured, solve pair on the 180k-node grid (against k_sptrsv.cu): 64 columns
// 1.06 ms (3.62), 16 columns 0.42 (1.51); 160,000 nodes in one layer, 4 columns
// 0.28 ms (0.32 with four warps everywhere); 40,000 nodes in four layers, 8
// columns 0.19 (0.23), 32 columns 0.28 (0.32); 57,600 nodes in four layers, 200
// columns 1.26 (4.3).  Below 32 columns the chain of 28 to 30 levels bounds it;
// at 64 columns the tensor pipe is busy a third of the time and the rest is the
// issue of splitting and conversion and the levels' last CTAs.  16 panel rows x
// 8 or 16 right-hand sides per warp (the panel as A operand) measured 1.48 and
// 1.58 ms at 64 columns; two row tiles per CTA on the narrow levels 0.20 ms for
// 0.19 at 8 columns; prefetching the operands of the next K step into
// registers, and the right-hand sides' addresses, nothing or a loss.
#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "split8.cuh"

namespace matex {

namespace {

using namespace s8;

constexpr int kMmRing = 4;   // panel tiles in a warp's ring, four warps
constexpr int kMmRing8 = 5;  // eight warps: a chunk's half of the K steps and one

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// store into the same variable of the cluster's CTA `rank`
__device__ __forceinline__ void st_cluster(const double* own, uint32_t rank, double v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(own)), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

// the two warps of pair p (of four)
__device__ __forceinline__ void pair_sync(int p) {
  asm volatile("bar.sync %0, 64;" ::"r"(p + 1) : "memory");
}

// Panel tiles of every supernode of one direction (setup).  A warp takes (row
// tile, chunk) pairs of supernode blockIdx.x; lane (g, t): row g, terms 2t,
// 2t + 1, 2t + 8, 2t + 9 of every K step, as mma.sync holds B.
__global__ void __launch_bounds__(256)
mm_split_kernel(const double* __restrict__ pan, const double* __restrict__ dinv,
                const MmSup* __restrict__ sups, const int32_t* __restrict__ klist, int fwd,
                unsigned char* __restrict__ A) {
  const MmSup d = sups[blockIdx.x];
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int rows = fwd ? d.ld : d.w, red = fwd ? d.w : d.ld;
  const int nch = (d.ks + kChunkSteps - 1) / kChunkSteps;
  const double* P = pan + d.pan;
  for (int it = blockIdx.y * 8 + (threadIdx.x >> 5); it < d.rt * nch; it += gridDim.y * 8) {
    const int rt = it / nch, ch = it - rt * nch;
    const int r = rt * 8 + g;
    const int ke = min(d.ks, (ch + 1) * kChunkSteps);
    auto val = [&](int k) {
      if (r >= rows || k >= red) return 0.0;
      // D^{-1} in the forward's y; the signs of -u_R and -x_R
      if (fwd) {
        const double v = P[(int64_t)k * d.ld + r];
        return r < d.w ? v * dinv[d.f + r] : -v;
      }
      const double v = P[(int64_t)r * d.ld + k];
      return k < d.w ? v : -v;
    };
    int m = 0;
    for (int ks = ch * kChunkSteps; ks < ke; ++ks)
      for (int u = 0; u < 4; ++u) m = max(m, exp_key(val(ks * 16 + 2 * t + (u & 1) + (u >> 1) * 8)));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    const int e = key_exp(m);
    const int node = klist[(int64_t)d.dl * 8 + r];
    for (int ks = ch * kChunkSteps; ks < ke; ++ks) {
      uint64_t u[4];
      for (int v = 0; v < 4; ++v) u[v] = digits(val(ks * 16 + 2 * t + (v & 1) + (v >> 1) * 8), e);
      uint32_t b[kDigits];
#pragma unroll
      for (int p = 0; p < kDigits; ++p) {
        b[p] = 0;
#pragma unroll
        for (int v = 0; v < 4; ++v) b[p] |= (uint32_t)((u[v] >> (8 * (6 - p))) & 0xff) << (8 * v);
      }
      unsigned char* tile = A + (d.a + (int64_t)rt * d.ks + ks) * kTileBytes;
      reinterpret_cast<uint4*>(tile)[lane] = make_uint4(b[0], b[1], b[2], b[3]);
      reinterpret_cast<uint2*>(tile + kTile45)[lane] = make_uint2(b[4], b[5]);
      reinterpret_cast<uint32_t*>(tile + kTile6)[lane] = b[6];
      if (t == 0) {
        reinterpret_cast<int16_t*>(tile + kTileE)[g] = (int16_t)e;
        reinterpret_cast<int32_t*>(tile + kTileDst)[g] = node;
      }
    }
  }
}

struct MmArgs {
  const int32_t* abort;     // set before the launch: the CTAs leave
  const MmTask* tasks;
  const int4* units;
  const int32_t* klist;
  const unsigned char* A;
  double* Y;
  double* Y2;
  int ldy, ncols, ncb;
  int nmulti, nsingle;      // tasks of more than one chunk come first
  int cluster;              // CTAs sharing a multi-chunk task
};

constexpr int kMmDigits = kChunkSteps * kFragBytes;  // digits of the right-hand sides
constexpr int kMmPair = 4 * 128 * (int)sizeof(double);  // sums of the pairs' second warps
constexpr int kMmSums = kMmRowsNarrow * 8 * kMmCols;  // results of a multi-chunk task
// this CTA's sums over its chunks, and what the warps of the cluster's CTAs send
// for its part of the results, from either half of their K steps
constexpr int kMmPart = (kMmSums + 2 * kMmSums) * (int)sizeof(double);

template <int W, bool kFwd>
__global__ void __launch_bounds__(W * 32, W > 4 ? 2 : 4) mm_level_kernel(const MmArgs a) {
  constexpr int S = W > 4 ? kMmRing8 : kMmRing;
  constexpr int kMmThreads = W * 32;
  constexpr int kItems = kChunkSteps / W;  // fragments per warp and chunk
  constexpr bool kPairs = W > 4;           // warps w and w + 4 share a row tile's K steps
  // [digits of the right-hand sides][a ring of S tiles per warp][sums over chunks]
  extern __shared__ __align__(16) unsigned char mm_smem[];
  __shared__ int cmax[kMmPack][kMmCols];
  __shared__ int4 units[kMmRowsWide];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int wrow = warp & 3, khalf = warp >> 2;
  // which task and column block (innermost: the blocks share the panel in L2);
  // clusters of multi-chunk tasks first, then one CTA per task
  const int cs = a.cluster, nmc = a.nmulti * a.ncb * cs;
  int bid = blockIdx.x, rank = 0;
  const bool multi = bid < nmc;
  if (multi) {
    rank = bid % cs;
    bid /= cs;
  } else {
    bid += a.nmulti * a.ncb - nmc;
  }
  const int task = bid / a.ncb, c0 = (bid - task * a.ncb) * kMmCols;
  if (task >= a.nmulti + a.nsingle) return;  // the grid is a multiple of the cluster size
  const bool shared = multi && cs > 1;  // the same in every CTA of a cluster
  const MmTask tk = a.tasks[task];
  if (threadIdx.x < tk.nu) units[threadIdx.x] = __ldg(a.units + tk.u0 + threadIdx.x);
  for (int i = threadIdx.x; i < kMmPack * kMmCols; i += kMmThreads) (&cmax[0][0])[i] = 0;
  unsigned char* ring = mm_smem + kMmDigits + warp * (S * kTileBytes);
  // sums over a multi-chunk task's chunks, each entry one thread's own
  double* pair = reinterpret_cast<double*>(mm_smem + kMmDigits + W * S * kTileBytes);
  double* part = pair + (kPairs ? kMmPair / 8 : 0);
  if (multi)
    for (int i = threadIdx.x; i < 3 * kMmSums; i += kMmThreads) part[i] = 0.0;
  __syncthreads();
  // Each CTA of a cluster adds up 1/cs of the task's results: the others write
  // theirs into its shared memory (recv: [CTA, half of its K steps][result]),
  // and after one barrier nobody's memory is needed but one's own.  This first
  // arrival says that recv is cleared.
  if (shared) cluster_arrive();
  double* recv = part + kMmSums;
  const int lg = shared ? 31 - __clz(kMmSums / cs) : 0;  // results per CTA, a power of two
  auto send = [&](int e, double x) {
    st_cluster(recv + ((2 * rank + khalf) << lg) + (e & ((1 << lg) - 1)), (uint32_t)(e >> lg), x);
  };
  // this CTA's K steps [ka, kz), in pieces that end where the chunks do (a
  // chunk has its own row exponents)
  int ka = tk.kbeg, kz = tk.kend;
  if (multi) mm_share(tk.kbeg, tk.kend, rank, cs, ka, kz);
  const int chb = ka / kChunkSteps, che = ka < kz ? (kz - 1) / kChunkSteps + 1 : chb;
  // ---- the warp's panel tiles, in the order it takes them ----------------------
  // unit: {first tile, K steps [kb, ke) of its supernode, first slot << 16 | supernode}
  // its share of a row tile's K steps
  auto own = [&](int& kb, int& ke) {
    if (!kPairs) return;
    const int mid = kb + (ke - kb + 1) / 2;
    if (khalf) kb = mid;
    else ke = mid;
  };
  int pch = chb, pu = wrow - 4, pks = 0, pke = 0, pslot = 0;
  const unsigned char* psrc = nullptr;
  auto fetch = [&]() {
    while (pks >= pke && pch < che) {
      pu += 4;
      if (pu >= tk.nu) {
        pu = wrow - 4;
        ++pch;
        continue;
      }
      const int4 un = units[pu];
      pks = max(un.y & 0xffff, max(ka, pch * kChunkSteps));
      pke = min(un.y >> 16, min(kz, (pch + 1) * kChunkSteps));
      if (pks < pke) own(pks, pke);
      psrc = a.A + (int64_t)(un.x + pks) * kTileBytes + lane * 16;
    }
    if (pch < che) {
      const uint32_t dst = smem_u32(ring + pslot * kTileBytes) + lane * 16;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(psrc) : "memory");
      if (lane < kTileBytes / 16 - 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512), "l"(psrc + 512)
                     : "memory");
      psrc += kTileBytes;
      ++pks;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    pslot = pslot + 1 == S ? 0 : pslot + 1;
  };
#pragma unroll
  for (int i = 0; i < S - 1; ++i) fetch();
  // rows of the right-hand sides that the first chunk's fragments take
  int rows[kItems][4];
  auto load_rows = [&](int k0, int k1) {
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int ks = k0 + warp + i * W;
      const int2* kl = reinterpret_cast<const int2*>(a.klist + (int64_t)(tk.kl + ks) * 16);
      int2 x = make_int2(-1, -1), y = x;
      if (ks < k1) {
        x = __ldg(kl + t);
        y = __ldg(kl + t + 4);
      }
      rows[i][0] = x.x;
      rows[i][1] = x.y;
      rows[i][2] = y.x;
      rows[i][3] = y.y;
    }
  };
  if (chb < che)
    load_rows(ka, min(kz, (chb + 1) * kChunkSteps));
  const bool direct = shared && che - chb == 1;  // results are sent as they are made
  if (shared) cluster_wait();  // every CTA's recv is cleared
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // uniform over the grid, looked at when the right-hand sides are on their way
  const bool stop = a.abort && __ldcg(a.abort);
  const bool upper = c0 + 8 < a.ncols;  // columns 8..15 of the block exist
  int slot = 0;
  for (int ch = chb; ch < che; ++ch) {
    const int k0 = max(ka, ch * kChunkSteps), k1 = min(kz, (ch + 1) * kChunkSteps);
    // ---- 1. the right-hand sides' digits: lane columns g and g + 8 -------------
    if (ch > chb) load_rows(k0, k1);
    double v[kItems][2][4];
#pragma unroll
    for (int i = 0; i < kItems; ++i)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = rows[i][u];
        const double* src = (!kFwd && (r & kMmAdd) == 0 ? a.Y2 : a.Y) +
                            (int64_t)(r & (kMmAdd - 1)) * a.ldy + c0 + g;
        v[i][0][u] = r >= 0 && c0 + g < a.ncols ? __ldcg(src) : 0.0;
        v[i][1][u] = r >= 0 && c0 + g + 8 < a.ncols ? __ldcg(src + 8) : 0.0;
      }
    if (stop) break;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int ks = k0 + warp + i * W;
      if (ks >= k1) continue;  // uniform over the warp
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h && !upper) break;
        int key = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) key = max(key, exp_key(v[i][h][u]));
        key = max(key, __shfl_xor_sync(0xffffffffu, key, 1));
        key = max(key, __shfl_xor_sync(0xffffffffu, key, 2));
        if (t == 0) atomicMax(&cmax[(tk.emap >> (4 * (ks & 7))) & 15][g + 8 * h], key);
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      const int ks = k0 + warp + i * W;
      if (ks >= k1) continue;
      const int* cm = cmax[(tk.emap >> (4 * (ks & 7))) & 15];
      uint32_t lo[2][kDigits], hi[2][kDigits];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h && !upper) {
#pragma unroll
          for (int p = 0; p < kDigits; ++p) lo[h][p] = hi[h][p] = 0;
          break;
        }
        const int e = key_exp(cm[g + 8 * h]);
        widen_pair(digits(v[i][h][0], e), digits(v[i][h][1], e), lo[h]);
        widen_pair(digits(v[i][h][2], e), digits(v[i][h][3], e), hi[h]);
      }
      uint4* fr = reinterpret_cast<uint4*>(mm_smem + (ks - k0) * kFragBytes) + lane;
#pragma unroll
      for (int p = 0; p < kDigits; ++p) fr[32 * p] = make_uint4(lo[0][p], lo[1][p], hi[0][p], hi[1][p]);
    }
    __syncthreads();
    // ---- 2. row tiles ----------------------------------------------------------
    for (int u = wrow; u < tk.nu; u += 4) {
      const int4 un = units[u];
      int kb = max(un.y & 0xffff, k0 - (un.z >> 16)), ke = min(un.y >> 16, k1 - (un.z >> 16));
      if (kb >= ke) continue;
      own(kb, ke);  // may leave the second warp of a pair none: its sums are zero
      const bool few = ke - kb <= 2;  // every sum below 2^22: no conversion afterwards
      float c[4][kDigits];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < kDigits; ++q) c[i][q] = few || q < 2 ? kBiasedZero : 0.f;
      int er[2], dst[2];
      const uint4* fr = reinterpret_cast<const uint4*>(mm_smem + ((un.z >> 16) + kb - k0) * kFragBytes) + lane;
      uint4 af[kDigits];
      uint32_t tp[kDigits];
      auto load = [&](int ks, uint4(&x)[kDigits], uint32_t(&y)[kDigits]) {
        // the tile has landed, and the warp is done with the one before it
        asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
        __syncwarp();
        fetch();
        const unsigned char* tile = ring + slot * kTileBytes;
        slot = slot + 1 == S ? 0 : slot + 1;
#pragma unroll
        for (int p = 0; p < kDigits; ++p) x[p] = fr[32 * p];
        fr += kFragBytes / 16;
        const uint4 t0 = reinterpret_cast<const uint4*>(tile)[lane];
        const uint2 t4 = reinterpret_cast<const uint2*>(tile + kTile45)[lane];
        y[0] = t0.x;
        y[1] = t0.y;
        y[2] = t0.z;
        y[3] = t0.w;
        y[4] = t4.x;
        y[5] = t4.y;
        y[6] = reinterpret_cast<const uint32_t*>(tile + kTile6)[lane];
        if (ks + 1 == ke) {
          const int e = reinterpret_cast<const int*>(tile + kTileE)[t];
          const int2 d = reinterpret_cast<const int2*>(tile + kTileDst)[t];
          er[0] = e & 0xffff;
          er[1] = e >> 16;
          dst[0] = d.x;
          dst[1] = d.y;
        }
      };
      auto multiply = [&](const uint4(&x)[kDigits], const uint32_t(&y)[kDigits]) {
#pragma unroll
        for (int p = 0; p < kDigits; ++p) {
          const uint32_t b0 = widen<0>(y[p]), b1 = widen<1>(y[p]);
#pragma unroll
          for (int r = 0; r + p < kDigits; ++r) mma(c, p + r, x[r], b0, b1);
          if (p > 0) mma(c, kDigits - 1, x[kDigits - p], down8(b0), down8(b1));
        }
      };
      for (int ks = kb; ks < ke; ++ks) {
        load(ks, af, tp);
        multiply(af, tp);
      }
      // ---- 3. FP64 values: columns g, g + 8 of panel rows 2t, 2t + 1 -------------
      double x[2][2] = {};
      if (!kPairs || kb < ke) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (h && !upper) break;
          const int key = cmax[un.z & 0xffff][g + 8 * h];
          const int ec = key >= kKeyInf ? kNonFinite : key_exp(key);
#pragma unroll
          for (int j = 0; j < 2; ++j)
            x[h][j] = few ? compose<true>(c[2 * h + j], er[j] + ec) : compose<false>(c[2 * h + j], er[j] + ec);
        }
      }
      if (direct) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (kb < ke && (k < 2 || upper)) send((u * 8 + 2 * t + (k & 1)) * kMmCols + g + 8 * (k >> 1), x[k >> 1][k & 1]);
        continue;
      }
      if constexpr (kPairs) {
        double* half = pair + wrow * 128 + lane;
        if (khalf)
#pragma unroll
          for (int k = 0; k < 4; ++k) half[32 * k] = x[k >> 1][k & 1];
        pair_sync(wrow);
        if (!khalf)
#pragma unroll
          for (int k = 0; k < 4; ++k) x[k >> 1][k & 1] += half[32 * k];
        if (u + 4 < tk.nu) pair_sync(wrow);
        if (khalf) continue;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h && !upper) break;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          if (multi) {
            part[(u * 8 + 2 * t + j) * kMmCols + g + 8 * h] += x[h][j];
          } else if (dst[j] >= 0 && c0 + g + 8 * h < a.ncols) {
            const int64_t o = (int64_t)(dst[j] & (kMmAdd - 1)) * a.ldy + c0 + g + 8 * h;
            if (!kFwd) a.Y[o] = x[h][j];
            else if (dst[j] & kMmAdd) atomicAdd(a.Y + o, x[h][j]);
            else a.Y2[o] = x[h][j];
          }
        }
      }
    }
    if (ch + 1 < che) {
      __syncthreads();  // every warp is done with this chunk's digits and exponents
      if (threadIdx.x < kMmCols) cmax[0][threadIdx.x] = 0;
      __syncthreads();
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (!multi || stop) return;
  const int nres = tk.nu * 8 * kMmCols;
  const int e0 = shared ? rank << lg : 0, ne = shared ? min(1 << lg, nres - e0) : nres;
  int dst[kMmSums / kMmThreads];
#pragma unroll
  for (int k = 0; k < kMmSums / kMmThreads; ++k) {
    const int i = threadIdx.x + k * kMmThreads;
    dst[k] = i < ne ? __ldg(a.klist + (int64_t)tk.dl * 8 + (e0 + i) / kMmCols) : -1;
  }
  if (!direct) __syncthreads();
  if (shared) {
    if (!direct && chb < che && khalf == 0)
      for (int e = threadIdx.x; e < nres; e += 4 * 32) send(e, part[e]);
    cluster_arrive();
    cluster_wait();
  }
#pragma unroll
  for (int k = 0; k < kMmSums / kMmThreads; ++k) {
    const int i = threadIdx.x + k * kMmThreads;
    if (i >= ne) break;
    const int col = c0 + (e0 + i) % kMmCols;
    if (dst[k] < 0 || col >= a.ncols) continue;
    double x;
    if (!shared) {
      x = part[i];
    } else {  // in a fixed order, pairs first
      double v[8];
#pragma unroll
      for (int r = 0; r < 8; ++r)
        v[r] = r >= cs ? 0.0 : kPairs ? recv[((2 * r) << lg) + i] + recv[((2 * r + 1) << lg) + i]
                                      : recv[((2 * r) << lg) + i];
      x = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    const int64_t o = (int64_t)(dst[k] & (kMmAdd - 1)) * a.ldy + col;
    if (!kFwd) a.Y[o] = x;
    else if (dst[k] & kMmAdd) atomicAdd(a.Y + o, x);
    else a.Y2[o] = x;
  }
}

template <int W>
constexpr int mm_smem_bytes(bool multi) {
  return kMmDigits + W * (W > 4 ? kMmRing8 : kMmRing) * kTileBytes + (W > 4 ? kMmPair : 0) +
         (multi ? kMmPart : 0);
}

template <int W, bool kFwd>
void launch_mm(const MmArgs& a, int grid, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)a.cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(W * 32);
  cfg.dynamicSmemBytes = mm_smem_bytes<W>(a.nmulti > 0);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = a.cluster > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, mm_level_kernel<W, kFwd>, a);
}

template <int W>
bool mm_limits() {
  return cudaFuncSetAttribute(mm_level_kernel<W, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              mm_smem_bytes<W>(true)) == cudaSuccess &&
         cudaFuncSetAttribute(mm_level_kernel<W, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              mm_smem_bytes<W>(true)) == cudaSuccess;
}

}  // namespace

bool mm_set_limits() { return mm_limits<8>() && mm_limits<4>(); }

size_t mm_tile_bytes() { return kTileBytes; }

void mm_split_panels(const double* pan, const double* dinv, const MmPlan& P, bool fwd,
                     unsigned char* A, cudaStream_t st) {
  if (P.nsup > 0)
    mm_split_kernel<<<dim3((unsigned)P.nsup, 8), 256, 0, st>>>(pan, dinv, P.sups[fwd ? 0 : 1],
                                                               P.klist[fwd ? 0 : 1], fwd ? 1 : 0, A);
}

int solve_mm(const int32_t* abort, const MmPlan& P, int fi, double* Y, double* Y2, int ldy, int ncols,
             cudaStream_t st) {
  int launches = 0;
  const int ncb = (ncols + kMmCols - 1) / kMmCols;
  for (int dir = 0; dir < 2; ++dir) {
    const bool fwd = dir == 0;
    for (int k = 0; k < P.nlev; ++k) {
      const int l = fwd ? k : P.nlev - 1 - k;
      // wide blocks of row tiles per CTA where the level fills the GPU with them
      const MmLevel& W = P.lev[dir][0][l];
      const MmLevel& N = P.lev[dir][1][l];
      const MmLevel& L = (long long)(W.nmulti + W.nsingle) * ncb >= kMmFill ? W : N;
      if (L.nmulti + L.nsingle == 0) continue;
      int cs = 1;
      while (cs < 8 && 4 * cs <= L.steps && (long long)L.nmulti * cs * ncb < kMmClusterFill) cs *= 2;
      const MmArgs a{abort, L.tasks, P.units[dir], P.klist[dir], P.A[fi][dir], Y, Y2, ldy,
                     ncols, ncb, L.nmulti, L.nsingle, cs};
      const int grid = L.nmulti * ncb * cs + (L.nsingle * ncb + cs - 1) / cs * cs;
      if (&L == &N && grid <= kMmDeep) {
        if (fwd) launch_mm<8, true>(a, grid, st);
        else launch_mm<8, false>(a, grid, st);
      } else {
        if (fwd) launch_mm<4, true>(a, grid, st);
        else launch_mm<4, false>(a, grid, st);
      }
      ++launches;
    }
  }
  return launches;
}

}  // namespace matex
