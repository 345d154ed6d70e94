// Krylov-side kernels of batched R-MATEX: segment inputs (Eq. 5/6), the start
// vector v = x(t) + F, Gram-Schmidt (two classical passes; Alg. 1 writes
// modified Gram-Schmidt, which CGS2 matches to rounding), the rational
// Hessenberg map H_m = (I - Htilde_m^{-1})/gamma (Eq. 9), the residual test of
// Sec. 3.3.3 and the coefficient vectors ||v|| e^{h H_m} e_1 at the output
// times of a segment (Alg. 2, "snapshots" reuse the basis).
#include "kernels.h"
#include "column_steps.cuh"

namespace matex {

namespace {

__global__ void input_rhs_kernel(double* __restrict__ Y, int ldy, int K, RoundCols rc,
                                 SourceTable src) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= K) return;
  const int g = rc.sgroup ? rc.sgroup[q] : rc.group[q];
  const double l0 = rc.l0[q], L = rc.len[q], l1 = l0 + L;
  for (int p = src.grp_ptr[g]; p < src.grp_ptr[g + 1]; ++p) {
    const int s = src.grp_src[p];
    const int o = src.pwl_off[s], np = src.pwl_off[s + 1] - o;
    const double u0 = pwl_eval(src.pwl_t + o, src.pwl_v + o, np, l0);
    const double val = (pwl_eval(src.pwl_t + o, src.pwl_v + o, np, l1) - u0) / L;
    Y[(int64_t)src.node[s] * ldy + q] += val;
  }
}

__global__ void advance_z_kernel(double* __restrict__ Z, const double* __restrict__ Zp,
                                 const double* __restrict__ X, int64_t gstride, RoundCols rc,
                                 int64_t n, double* __restrict__ pbound) {
  const int q = blockIdx.y;
  if (blockIdx.x == 0 && threadIdx.x < 2) pbound[2 * q + threadIdx.x] = 0.0;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t g = rc.group[q];
  const int64_t k = g * gstride + i;
  if (rc.seg[q] == 0) Z[k] = X[k];
  else Z[k] = fma(rc.lprev[q], Zp[k], Z[k]);
}

__global__ void initial_rhs_kernel(double* __restrict__ Y, int ldy, int K, SourceTable src,
                                   const int32_t* __restrict__ groups) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= K) return;
  const int g = groups[q];
  for (int p = src.grp_ptr[g]; p < src.grp_ptr[g + 1]; ++p) {
    const int s = src.grp_src[p];
    const int o = src.pwl_off[s], np = src.pwl_off[s + 1] - o;
    Y[(int64_t)src.node[s] * ldy + q] += pwl_eval(src.pwl_t + o, src.pwl_v + o, np, 0.0);
  }
}

constexpr int kRedThreads = 256;

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  return s;  // valid in thread 0
}

__global__ void __launch_bounds__(kRedThreads)
krylov_start_kernel(double* __restrict__ Vb, int64_t vstride, const double* __restrict__ X,
                    const double* __restrict__ Z, const double* __restrict__ Zp,
                    const double* __restrict__ W, unsigned long long* __restrict__ pbound,
                    int64_t gstride, const int32_t* __restrict__ groups,
                    const int32_t* __restrict__ vslots, int64_t n, double* __restrict__ partials,
                    int nchunks) {
  __shared__ double red[32];
  const int q = blockIdx.y;
  const int64_t g = groups[q];
  const int64_t vs = vslots[q];
  const int64_t b = (int64_t)blockIdx.x * kChunk;
  const int64_t e = min(n, b + kChunk);
  double acc = 0.0;
  // |w - z| and |z'| are >= 0 (or NaN without its sign bit): their bit patterns
  // order like the values, a NaN above +inf
  unsigned long long pa = 0, pb = 0;
  constexpr unsigned long long kAbs = 0x7fffffffffffffffull;
  for (int64_t i = b + threadIdx.x; i < e; i += blockDim.x) {
    const double wz = W[g * gstride + i] - Z[g * gstride + i];
    const double v = X[g * gstride + i] + wz;
    Vb[vs * vstride + i] = v;
    acc = fma(v, v, acc);
    pa = max(pa, (unsigned long long)__double_as_longlong(wz) & kAbs);
    pb = max(pb, (unsigned long long)__double_as_longlong(Zp[g * gstride + i]) & kAbs);
  }
  for (int off = 16; off > 0; off >>= 1) {
    pa = max(pa, __shfl_xor_sync(0xffffffffu, pa, off));
    pb = max(pb, __shfl_xor_sync(0xffffffffu, pb, off));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(pbound + 2 * q, pa);
    atomicMax(pbound + 2 * q + 1, pb);
  }
  const double s = block_sum(acc, red);
  if (threadIdx.x == 0) partials[(int64_t)q * nchunks + blockIdx.x] = s;
}

__global__ void basis_scale_kernel(double* __restrict__ Vb, int64_t vstride,
                                   const int32_t* __restrict__ groups,
                                   const int32_t* __restrict__ iter, int wslot,
                                   const double* __restrict__ scale, int64_t n) {
  const int q = iter[blockIdx.y];
  const int64_t g = groups[q];
  const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= n) return;
  Vb[g * vstride + (int64_t)wslot * n + x] *= scale[q];
}

// The columns p < K_in (list iter_in, or all in order) with status 0, kept in
// order in iter_out with their slots in iter_grp, their number in *count, by
// one CTA.  With expected >= 0 (a recorded run, whose launches were sized for
// that many) another number raises ca.flag and points the surplus entries at
// column 0, so that the rest of the replay, whose result is discarded, stays in
// range.
__device__ void compact_columns(SmallState ss, const CompactArgs& ca, const int32_t* iter_in, int K_in) {
  __shared__ int warp_cnt[33];
  __shared__ int base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  if (threadIdx.x == 0) base = 0;
  for (int p0 = 0; p0 < K_in; p0 += blockDim.x) {
    const int p = p0 + (int)threadIdx.x;
    const int q = p < K_in ? (iter_in ? iter_in[p] : p) : 0;
    const bool live = p < K_in && __ldcg(ss.status + q) == 0;
    const unsigned mask = __ballot_sync(0xffffffffu, live);
    if (lane == 0) warp_cnt[warp] = __popc(mask);
    __syncthreads();
    if (threadIdx.x == 0) {
      int s = base;
      for (int w = 0; w < nw; ++w) {
        const int c = warp_cnt[w];
        warp_cnt[w] = s;
        s += c;
      }
      base = s;
    }
    __syncthreads();
    if (live) {
      const int k = warp_cnt[warp] + __popc(mask & ((1u << lane) - 1u));
      ca.iter_grp[k] = ca.slots[q];
      ca.iter_out[k] = q;
    }
    __syncthreads();
  }
  const int cnt = base;
  if (threadIdx.x == 0) {
    *ca.count = cnt;
    if (ca.expected >= 0 && cnt != ca.expected) *ca.flag = 1;
  }
  if (ca.expected > cnt)
    for (int k = cnt + (int)threadIdx.x; k < ca.expected; k += blockDim.x) {
      ca.iter_out[k] = 0;
      ca.iter_grp[k] = ca.slots[0];
    }
}

// True in the CTA of the grid that arrives last, whose threads then see what
// the others wrote; the counter is zero again afterwards.
__device__ bool last_cta(int32_t* arrived) {
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(arrived, 1) == (int)gridDim.x - 1;
    if (last) *arrived = 0;
    __threadfence();
  }
  __syncthreads();
  return last != 0;
}

__global__ void __launch_bounds__(kRedThreads)
start_finish_kernel(const double* __restrict__ partials, int nchunks, int K, SmallState ss,
                    CompactArgs ca) {
  __shared__ double red[32];
  const int c = blockIdx.x;
  double acc = 0.0;
  for (int k = threadIdx.x; k < nchunks; k += blockDim.x) acc += partials[(int64_t)c * nchunks + k];
  const double s = block_sum(acc, red);
  for (int i = threadIdx.x; i < kMaxB * kMaxM; i += blockDim.x) ss.Ht[(int64_t)c * kMaxB * kMaxM + i] = 0.0;
  if (threadIdx.x == 0) {
    const double beta = sqrt(s);
    ss.beta[c] = beta;
    ss.m[c] = 0;
    const bool quiet = beta <= 1e-300;
    ss.status[c] = quiet ? 4 : 0;
    ss.scale[c] = quiet ? 0.0 : 1.0 / beta;
  }
  if (last_cta(ca.arrived)) compact_columns(ss, ca, nullptr, K);
}

__global__ void __launch_bounds__(kTeamThreads)
residual_kernel(SmallState ss, RoundCols rc, const int32_t* __restrict__ iter, int j, double gamma,
                double tol, int m_max, const int32_t* __restrict__ replay, CompactArgs ca) {
  extern __shared__ double smem_raw[];
  SmallShared<CtaTeam::kWorkers>& sh = *reinterpret_cast<SmallShared<CtaTeam::kWorkers>*>(smem_raw);
  residual_column<CtaTeam>(ss, rc, iter[blockIdx.x], j, gamma, tol, m_max, replay, 0.0, sh);
  if (last_cta(ca.arrived)) compact_columns(ss, ca, iter, gridDim.x);
}

__global__ void record_kernel(SmallState ss, RoundCols rc, int K, int32_t* m_rec, int32_t* st_rec) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= K) return;
  m_rec[rc.segid[q]] = ss.m[q];
  st_rec[rc.segid[q]] = ss.status[q];
}

__global__ void __launch_bounds__(kTeamThreads)
coef_kernel(SmallState ss, RoundCols rc, double gamma, double dt_out, double* __restrict__ coef,
            int ldo, double* __restrict__ yend, double tail_eps, const double* __restrict__ pbound,
            int32_t* __restrict__ tcut) {
  extern __shared__ double smem_raw[];
  SmallShared<CtaTeam::kWorkers>& sh = *reinterpret_cast<SmallShared<CtaTeam::kWorkers>*>(smem_raw);
  if (threadIdx.x == 0) sh.cm = 0;  // no residual test ran in this CTA
  __syncthreads();
  coef_column<CtaTeam>(ss, rc, blockIdx.x, gamma, dt_out, coef, ldo, yend, tail_eps, pbound, tcut, sh);
}

// One matrix per CTA: 64 threads up to 8 x 8 (an entry each), 128 beyond.
__global__ void __launch_bounds__(kSmallThreads)
expm_batch_kernel(int m, const double* __restrict__ A, const double* __restrict__ h,
                  double* __restrict__ E) {
  __shared__ ExpmWork w;
  __shared__ double H[kMat];
  const int b = blockIdx.x;
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) H[(e / m) * kLd + e % m] = A[(int64_t)b * m * m + e];
  __syncthreads();
  expm_dev(H, h[b], H, m, w);
  for (int e = threadIdx.x; e < m * m; e += blockDim.x) E[(int64_t)b * m * m + e] = H[(e / m) * kLd + e % m];
}

}  // namespace

void build_input_rhs(double* Y, int ldy, int K, const RoundCols& rc, const SourceTable& src,
                     int64_t n, cudaStream_t st) {
  cudaMemsetAsync(Y, 0, sizeof(double) * (size_t)n * ldy, st);
  input_rhs_kernel<<<(K + 127) / 128, 128, 0, st>>>(Y, ldy, K, rc, src);
}

void advance_z(double* Z, const double* Zp, const double* X, int64_t gstride, const RoundCols& rc,
               int K, int64_t n, double* pbound, cudaStream_t st) {
  if (K <= 0) return;
  dim3 grid((unsigned)((n + 255) / 256), (unsigned)K);
  advance_z_kernel<<<grid, 256, 0, st>>>(Z, Zp, X, gstride, rc, n, pbound);
}

void build_initial_rhs(double* Y, int ldy, int K, const SourceTable& src, const int32_t* groups,
                       int64_t n, cudaStream_t st) {
  cudaMemsetAsync(Y, 0, sizeof(double) * (size_t)n * ldy, st);
  initial_rhs_kernel<<<(K + 127) / 128, 128, 0, st>>>(Y, ldy, K, src, groups);
}

void krylov_start(double* Vbase, int64_t vstride, const double* X, const double* Z, const double* Zp,
                  const double* W, double* pbound, int64_t gstride, const int32_t* groups, const int32_t* vslots, int K, int64_t n,
                  double* partials, int nchunks, cudaStream_t st) {
  dim3 grid((unsigned)nchunks, (unsigned)K);
  krylov_start_kernel<<<grid, kRedThreads, 0, st>>>(
      Vbase, vstride, X, Z, Zp, W, reinterpret_cast<unsigned long long*>(pbound), gstride, groups,
      vslots, n, partials, nchunks);
}

void basis_scale(double* Vbase, int64_t vstride, const int32_t* groups, const int32_t* iter, int K,
                 int wslot, const double* scale, int64_t n, cudaStream_t st) {
  dim3 grid((unsigned)((n + 255) / 256), (unsigned)K);
  basis_scale_kernel<<<grid, 256, 0, st>>>(Vbase, vstride, groups, iter, wslot, scale, n);
}

void start_finish(const double* partials, int nchunks, int K, SmallState ss, const CompactArgs& ca,
                  cudaStream_t st) {
  start_finish_kernel<<<K, kRedThreads, 0, st>>>(partials, nchunks, K, ss, ca);
}

namespace {
__global__ void apply_A_kernel(double* __restrict__ Vb, int64_t vstride,
                               const int32_t* __restrict__ iter_grp, int jsrc, int jdst,
                               const int64_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                               const double* __restrict__ val, const double* __restrict__ c,
                               int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double* __restrict__ v = Vb + (int64_t)iter_grp[blockIdx.y] * vstride + (int64_t)jsrc * n;
  double gv = 0.0;
  for (int64_t k = rowptr[i]; k < rowptr[i + 1]; ++k) gv = fma(val[k], v[col[k]], gv);
  Vb[(int64_t)iter_grp[blockIdx.y] * vstride + (int64_t)jdst * n + i] = -gv / c[i];
}

}  // namespace

void krylov_apply_A(double* Vb, int64_t vstride, const int32_t* iter_grp, int K, int jsrc, int jdst,
                    const int64_t* rowptr, const int32_t* col, const double* val, const double* c,
                    int64_t n, cudaStream_t st) {
  if (K <= 0) return;
  dim3 grid((unsigned)((n + 255) / 256), (unsigned)K);
  apply_A_kernel<<<grid, 256, 0, st>>>(Vb, vstride, iter_grp, jsrc, jdst, rowptr, col, val, c, n);
}

void residual_check(SmallState ss, const RoundCols& rc, int K, int j, double gamma, double tol,
                    int m_max, const int32_t* replay, const int32_t* iter_in, const CompactArgs& ca,
                    cudaStream_t st) {
  residual_kernel<<<K, kTeamThreads, sizeof(SmallShared<CtaTeam::kWorkers>), st>>>(
      ss, rc, iter_in, j, gamma, tol, m_max, replay, ca);
}

void record_segments(const SmallState& ss, const RoundCols& rc, int K, int32_t* m_rec,
                     int32_t* st_rec, cudaStream_t st) {
  if (K <= 0) return;
  record_kernel<<<(K + 127) / 128, 128, 0, st>>>(ss, rc, K, m_rec, st_rec);
}

void output_coefficients(SmallState ss, const RoundCols& rc, int K, double gamma, double dt_out,
                         double* coef, int ldo, double* yend, cudaStream_t st, double tail_eps,
                         const double* pbound, int32_t* tcut) {
  coef_kernel<<<K, kTeamThreads, sizeof(SmallShared<CtaTeam::kWorkers>), st>>>(
      ss, rc, gamma, dt_out, coef, ldo, yend, tail_eps, pbound, tcut);
}

void expm_batch(int batch, int m, const double* A, const double* h, double* E, cudaStream_t st) {
  expm_batch_kernel<<<batch, m <= 8 ? 64 : kSmallThreads, 0, st>>>(m, A, h, E);
}

void set_small_smem_limits() {
  const int bytes = (int)sizeof(SmallShared<CtaTeam::kWorkers>);
  cudaFuncSetAttribute(residual_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  cudaFuncSetAttribute(coef_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace matex
