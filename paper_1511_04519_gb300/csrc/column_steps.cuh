// Per-column small steps of one segment, executed by a team of threads (a CTA,
// or the first warps of one): the residual test of Sec. 3.3.3 after Arnoldi step j, and
// the coefficient vectors ||v|| e^{h H_m} e_1 at the segment's outputs and its
// end (Alg. 2, "snapshots" reuse the basis).  Shared by the batched kernels
// (one CTA per column of a round) and the resident round kernel (one CTA runs
// a column's whole segment).
#pragma once
#include "kernels.h"
#include "small_dense.cuh"

namespace matex {
namespace {

using ExpmWork = SmallWork<kMaxM>;
constexpr int kLd = Small<kMaxM>::kLd;
constexpr int kMat = Small<kMaxM>::kMat;

template <class G = CtaGroup>
__device__ __forceinline__ void expm_dev(const double* M, double h, double* E, int m, ExpmWork& w) {
  Small<kMaxM, G>::expm(M, h, E, m, w);
}
template <class G = CtaGroup>
__device__ __forceinline__ void rational_H(const double* Ht, int m, double gamma, double* H,
                                           ExpmWork& w, int variant) {
  Small<kMaxM, G>::rational_H(Ht, m, gamma, H, w, variant);
}

// value at x of the piecewise-linear source (t, v) with np breakpoints, held
// constant outside [t_0, t_{np-1}]
__device__ __forceinline__ double pwl_eval(const double* t, const double* v, int np, double x) {
  if (x <= t[0]) return v[0];
  if (x >= t[np - 1]) return v[np - 1];
  int j = 0;
  while (j + 1 < np && t[j + 1] <= x) ++j;
  const double slope = (v[j + 1] - v[j]) / (t[j + 1] - t[j]);
  return slope * (x - t[j]) + v[j];
}

// How the threads of a call share the small steps: kWorkers groups W run
// independent exponentials at once, G (all of the call's threads) the rest.
struct CtaTeam {  // the batched kernels: a CTA of three groups of 64 threads
  using G = CtaGroup;
  using W = WorkGroup;
  static constexpr int kWorkers = kTeamThreads / kWorkThreads;
  static __device__ __forceinline__ int worker() { return threadIdx.x / kWorkThreads; }
};
struct WarpTeam {  // the resident rounds: the first three warps of the CTA
  struct G {
    static __device__ __forceinline__ int rank() { return threadIdx.x; }
    static __device__ __forceinline__ int size() { return 96; }
    static __device__ __forceinline__ void sync() { asm volatile("bar.sync 1, 96;" ::: "memory"); }
  };
  using W = WarpGroup;
  static constexpr int kWorkers = 3;
  static __device__ __forceinline__ int worker() { return threadIdx.x / 32; }
};
struct WarpSolo {  // the resident rounds where three work areas do not fit
  using G = WarpGroup;
  using W = WarpGroup;
  static constexpr int kWorkers = 1;
  static __device__ __forceinline__ int worker() { return 0; }
};

template <int NW>
struct SmallShared {
  ExpmWork w[NW];
  double H[kMat];
  double y[kMaxM];
  int flag, last;
  // H of Krylov dimension cm and exponentials e^{ch[i] H} (ce[i]): at the
  // segment's first output, its end and one output interval; cm = 0: none.  The
  // caller clears cm where the shared memory is not that of the test's own CTA.
  int cm;
  double ch[3];
  double ce[3][kMat];
};

// e^{hH} at h = t[k] into sh.ce[k] for the k in want[0..count), one worker each
template <class Team>
__device__ void team_expm(const double (&t)[3], const int (&want)[3], int count, int m,
                          SmallShared<Team::kWorkers>& sh) {
  for (int i = Team::worker(); i < count; i += Team::kWorkers)
    expm_dev<typename Team::W>(sh.H, t[want[i]], sh.ce[want[i]], m, sh.w[Team::worker()]);
  Team::G::sync();
}

// Status of column q after Arnoldi step j (m = j + 1), returned to every
// thread and stored in ss.status[q]: 0 iterate on, 1 converged (or the
// replayed dimension reached), 2 happy breakdown, 3 m_max reached unconverged.
// The residual of Sec. 3.3.3, ||v|| |h_{m+1,m} e_m^T e^{hH} e_1| (h_{m+1,m}
// scaled by ss.rscale), is taken at the segment's first output and at its end.
// With dt > 0 an idle worker also takes e^{dt H}, which the coefficients of a
// converged column need.  Ht and ss.beta[q] may have been written by any thread
// of the CTA before the call.
template <class Team>
__device__ int residual_column(SmallState ss, const RoundCols& rc, int q, int j, double gamma,
                               double tol, int m_max, const int32_t* __restrict__ replay, double dt,
                               SmallShared<Team::kWorkers>& sh) {
  using G = typename Team::G;
  const int m = j + 1;
  const double* Ht = ss.Ht + (int64_t)q * kMaxB * kMaxM;
  G::sync();  // Ht complete; sh.flag of an earlier call has been read
  if (G::rank() == 0) {
    const double hnext = Ht[m * kMaxM + (m - 1)];
    ss.m[q] = m;
    int st = 0;
    if (hnext <= 1e-13 * fabs(Ht[0])) st = 2;  // happy breakdown (h_11 < 0 for A itself)
    else if (replay) st = (replay[rc.segid[q]] <= m) ? 1 : 0;
    sh.flag = st;
    sh.cm = 0;
  }
  G::sync();
  int st = sh.flag;
  if (st == 0 && !replay) {
    rational_H<G>(Ht, m, gamma, sh.H, sh.w[0], ss.krylov);
    const double L = rc.len[q];
    const double t[3] = {fmin(rc.hfirst[q], L), L, dt};
    const int all[3] = {0, 1, 2};
    team_expm<Team>(t, all, dt > 0.0 && Team::kWorkers > 2 ? 3 : 2, m, sh);
    if (G::rank() == 0) {
      // r = ||v|| |s h_{m+1,m} e_m^T e^{hH} e_1|, s making h_{m+1,m} dimensionless
      const double c = ss.beta[q] * fabs(ss.rscale * Ht[m * kMaxM + (m - 1)]);
      const double rmax = fmax(c * fabs(sh.ce[0][(m - 1) * kLd]), c * fabs(sh.ce[1][(m - 1) * kLd]));
      sh.flag = rmax < tol ? 1 : 0;
      sh.cm = m;
      sh.ch[0] = t[0];
      sh.ch[1] = L;
      sh.ch[2] = dt > 0.0 && Team::kWorkers > 2 ? dt : -1.0;
    }
    G::sync();
    st = sh.flag;
  }
  if (st == 0 && m >= m_max) st = 3;
  if (G::rank() == 0) ss.status[q] = st;
  return st;
}

// Coefficients of column q at the outputs of its segment: coef row o holds
// y(h_o) = ||v|| e^{h_o H_m} e_1 (h_o = t_o - l_j) in slots 0..m-1 and h_o in
// slot kMaxM; yend[q] = y(L).  With tail_eps > 0 and pbound given, tcut[q]
// receives the tail cut (outputs up to the last one whose ||y||_2 exceeds
// tail_eps/2 keep V y; a NaN norm or bound counts as large).  The outputs are
// equally spaced: with those of [0, B) known, e^{B dt H} gives [B, 2B) at once
// (a chain of ten squarings for a thousand outputs, where one output after the
// other took 190 us).
template <class Team>
__device__ void coef_column(SmallState ss, const RoundCols& rc, int q, double gamma, double dt_out,
                            double* __restrict__ coef, int ldo, double* __restrict__ yend,
                            double tail_eps, const double* __restrict__ pbound,
                            int32_t* __restrict__ tcut, SmallShared<Team::kWorkers>& sh) {
  using G = typename Team::G;
  const int m = ss.m[q];
  const int no = rc.nout[q];
  double* cq = coef + (int64_t)q * ldo * kCoefLd;
  const bool cut = pbound != nullptr && tail_eps > 0.0;
  if (G::rank() == 0) sh.last = -1;
  // step of the -P term at every output: h = t_o - l_j with t_o = o * dt_out
  for (int o = G::rank(); o < no; o += G::size())
    cq[(int64_t)o * kCoefLd + kMaxM] = (double)(rc.obeg[q] + o) * dt_out - rc.l0[q];
  if (m > 0) {
    const double* Ht = ss.Ht + (int64_t)q * kMaxB * kMaxM;
    const double beta = ss.beta[q];
    const double hf = rc.hfirst[q], L = rc.len[q];
    // at the first output, the segment's end and the output interval, without
    // those that the residual test of this m took
    const bool have = sh.cm == m;
    const double t[3] = {hf, L, dt_out};
    int want[3], count = 0;
    if (no > 0 && !(have && sh.ch[0] == hf)) want[count++] = 0;
    if (!(have && sh.ch[1] == L)) want[count++] = 1;
    if (no > 1 && !(have && sh.ch[2] == dt_out)) want[count++] = 2;
    if (!have) rational_H<G>(Ht, m, gamma, sh.H, sh.w[0], ss.krylov);
    team_expm<Team>(t, want, count, m, sh);
    for (int i = G::rank(); i < m; i += G::size()) {
      yend[(int64_t)q * kMaxM + i] = beta * sh.ce[1][i * kLd];
      if (no > 0) cq[i] = beta * sh.ce[0][i * kLd];
    }
    G::sync();
    double *P = sh.ce[2], *Q = sh.ce[0];
    for (int B = 1; B < no; B *= 2) {
      const int cnt = min(B, no - B);
      for (int e = G::rank(); e < cnt * m; e += G::size()) {
        const int o = e / m, i = e - o * m;
        const double* y = cq + (int64_t)o * kCoefLd;
        double s = 0.0;
        for (int k = 0; k < m; ++k) s = fma(P[i * kLd + k], y[k], s);
        cq[(int64_t)(B + o) * kCoefLd + i] = s;
      }
      if (2 * B < no) {
        Small<kMaxM, G>::mat_mul(P, P, Q, m);
        double* t = P; P = Q; Q = t;
      } else {
        G::sync();
      }
    }
    if (cut) {
      const double e2 = 0.25 * tail_eps * tail_eps;
      for (int o = G::rank(); o < no; o += G::size()) {
        const double* y = cq + (int64_t)o * kCoefLd;
        double s = 0.0;
        for (int k = 0; k < m; ++k) s = fma(y[k], y[k], s);
        if (!(s <= e2)) atomicMax(&sh.last, o);
      }
    }
  }
  G::sync();
  if (tcut != nullptr && G::rank() == 0) {
    tcut[2 * q] = cut ? sh.last + 1 : no;
    tcut[2 * q + 1] =
        cut && pbound[2 * q] + rc.len[q] * pbound[2 * q + 1] <= 0.5 * tail_eps ? 1 : 0;
  }
}

}  // namespace
}  // namespace matex
