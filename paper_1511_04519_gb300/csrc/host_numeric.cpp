// Host setup, part 2: numeric supernodal L D L^T by the multifrontal method.
// This is the one-time serial factorisation of Alg. 2 (UMFPACK's LU in the
// paper); the matrices are SPD here (C diagonal positive, G a grounded
// conductance matrix), so a symmetric factorisation without pivoting is used,
// for diagonally dominant ones without cancellation in the pivots.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <thread>

#include "internal.h"

namespace matex {

namespace {

// Run f(lo, hi) over [0, n) split across the host's cores (serially when
// `work` is small).
template <typename F>
void parallel_for(int64_t n, double work, F f) {
  int nt = (int)std::min<unsigned>(std::max(1u, std::thread::hardware_concurrency()), 32u);
  if (work < 4e6 || n < nt) nt = 1;
  if (nt == 1) {
    f((int64_t)0, n);
    return;
  }
  std::vector<std::thread> th;
  const int64_t chunk = (n + nt - 1) / nt;
  for (int t = 0; t < nt; ++t) {
    const int64_t lo = t * chunk, hi = std::min(n, lo + chunk);
    if (lo >= hi) break;
    th.emplace_back([=, &f] { f(lo, hi); });
  }
  for (auto& x : th) x.join();
}

// What every row of diag(dshift) + a sums to (a: the entries of A times alpha),
// for a diagonally dominant matrix without positive off-diagonal entries: grounded
// conductances and capacitances (dominant to 2^-40 of the diagonal, whose own
// rounding may miss it).  False for any other matrix.  The sums cancel, so their
// rounding errors are summed beside them (Knuth's two-sum; a comes as an array so
// that no compiler fuses its products into the sums).
bool row_excess(const CsrSym& A, const double* dshift, const std::vector<double>& a,
                std::vector<double>& ex) {
  ex.assign(A.n, 0.0);
  for (int64_t i = 0; i < A.n; ++i) {
    double s = dshift ? dshift[i] : 0.0, low = 0.0, diag = s;
    for (int64_t p = A.rowptr[i]; p < A.rowptr[i + 1]; ++p) {
      if (A.col[p] == i) diag += a[p];
      else if (!(a[p] <= 0.0)) return false;
      const double t = s + a[p], b = t - s;
      low += (s - (t - b)) + (a[p] - b);
      s = t;
    }
    ex[i] = s + low;
    if (!(ex[i] >= -0x1p-40 * diag)) return false;
  }
  return true;
}

// Sum of x[0..n) of one sign, in eight strands and halves: a rounding or two.
double even_sum(const double* x, int64_t n) {
  if (n > 512) {
    const int64_t h = n / 2 & ~(int64_t)7;
    return even_sum(x, h) + even_sum(x + h, n - h);
  }
  double s[8] = {};
  int64_t i = 0;
  for (; i + 8 <= n; i += 8)
    for (int k = 0; k < 8; ++k) s[k] += x[i + k];
  for (; i < n; ++i) s[i & 7] += x[i];
  return ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

constexpr int64_t kPanel = 64;

// Partial L D L^T of the first w columns of the front F (nr x nr, column-major,
// lower triangle): blocked right-looking, panels of 64 columns, the trailing
// update of each panel spread over threads (columns are independent).
// On return column j < w holds l_j (unit diagonal implied) below the diagonal
// and dinv[j] = 1/d_j; the trailing (nr-w) x (nr-w) block holds the Schur
// complement.  Returns false on a non-positive pivot.
// With v, the row sums of a matrix that row_excess accepts, the pivots are taken
// from them, d_j = v_j - sum_{i > j} f_ij, and v is carried along, v_i -= l_ij v_j
// (on return the Schur complement's row sums): everything then adds up values of
// one sign, where the diagonal f_jj minus its updates cancels down to what the
// grid's few grounded nodes leave (Grassmann, Taksar and Heyman, Oper. Res. 33,
// 1985; O'Cinneide, Numer. Math. 73, 1996).  Relative error of the solutions,
// root mean square over grids of 1,024 to 39,711 nodes in one to four layers:
// 2e-16 to 4.5e-16 instead of 1.7e-15 to 4.2e-15.
bool partial_ldlt(double* F, int64_t nr, int64_t w, double* dinv, std::vector<double>& W, double* v) {
  for (int64_t jb = 0; jb < w; jb += kPanel) {
    const int64_t b = std::min(kPanel, w - jb);
    // unscaled copies l_i d_j of the panel's columns, kept for the trailing update
    W.assign((size_t)b * nr, 0.0);
    for (int64_t j = jb; j < jb + b; ++j) {
      double* cj = &F[j * nr];
      const double d = v ? v[j] - even_sum(cj + j + 1, nr - j - 1) : cj[j];
      if (!(d > 0.0) || !std::isfinite(d)) return false;
      const double di = 1.0 / d;
      dinv[j] = di;
      double* wj = &W[(j - jb) * nr];
      for (int64_t i = j + 1; i < nr; ++i) wj[i] = cj[i];
      for (int64_t i = j + 1; i < nr; ++i) cj[i] *= di;
      if (v)
        for (int64_t i = j + 1; i < nr; ++i) v[i] -= cj[i] * v[j];
      // update the rest of the panel
      for (int64_t k = j + 1; k < jb + b; ++k) {
        const double lk = cj[k];
        if (lk == 0.0) continue;
        double* ck = &F[k * nr];
        for (int64_t i = k; i < nr; ++i) ck[i] -= wj[i] * lk;
      }
    }
    // trailing update: F[i][k] -= sum_j W[i][j] l_k,j for k >= jb+b, i >= k;
    // columns dealt cyclically over threads (the triangle shortens with k)
    const int64_t k0 = jb + b;
    const double work = (double)b * (double)(nr - k0) * (double)(nr - k0) / 2.0;
    const int64_t nt = std::max<int64_t>(1, std::min<int64_t>(32, std::thread::hardware_concurrency()));
    parallel_for(nt, work, [&](int64_t tlo, int64_t thi) {
      for (int64_t t = tlo; t < thi; ++t)
        for (int64_t kk = t; kk < nr - k0; kk += nt) {
          const int64_t k = k0 + kk;
          double* ck = &F[k * nr];
          for (int64_t j = jb; j < jb + b; ++j) {
            const double lk = F[j * nr + k];
            if (lk == 0.0) continue;
            const double* wj = &W[(j - jb) * nr];
            for (int64_t i = k; i < nr; ++i) ck[i] -= wj[i] * lk;
          }
        }
    });
  }
  return true;
}

}  // namespace

// Column k of the panel [L_ss^{-1}; L_Rs L_ss^{-1}] of the supernode at
// columns j0 .. j0 + w of the front (leading dimension nr), whose rows below
// are the front's rows at[0 .. r): x[0 .. w) by forward substitution on e_k,
// x[w .. w + r) = L_Rs x[0 .. w).  at = null: the rows right below the columns.
void panel_column(const double* front, int64_t nr, int64_t j0, int64_t w, int64_t r,
                  const int32_t* at, int64_t k, double* x) {
  x[k] = 1.0;
  for (int64_t j = k; j < w; ++j) {
    const double xj = x[j];
    if (xj == 0.0) continue;
    const double* cj = &front[(j0 + j) * nr];
    for (int64_t i = j + 1; i < w; ++i) x[i] -= cj[j0 + i] * xj;
    if (at)
      for (int64_t i = 0; i < r; ++i) x[w + i] += cj[at[i]] * xj;
    else
      for (int64_t i = 0; i < r; ++i) x[w + i] += cj[j0 + w + i] * xj;
  }
}

std::string numeric_ldlt(const CsrSym& A, const double* dshift, double alpha,
                         const Symbolic& S, Numeric& F, const Symbolic* coarse,
                         std::vector<double>* coarse_pan) {
  // the elimination runs on the coarse structure when there is one (larger
  // fronts, fewer extend-adds); S's panels are cut from its columns of L
  const Symbolic& T = coarse ? *coarse : S;
  const int64_t n = S.n;
  F.dinv.assign(n, 0.0);
  F.pan_cm.assign(S.pan_off[S.nsup], 0.0);
  F.pan_rm.assign(S.pan_off[S.nsup], 0.0);
  if (coarse_pan) coarse_pan->assign(T.pan_off[T.nsup], 0.0);
  std::vector<int32_t> pos(n, -1);
  std::vector<std::vector<double>> upd(T.nsup);
  std::vector<std::vector<int32_t>> kids(T.nsup);
  for (int32_t s = 0; s < T.nsup; ++s)
    if (T.sup_parent[s] >= 0) kids[T.sup_parent[s]].push_back(s);
  std::vector<double> front, lcol, excess, v;
  std::vector<double> scaled(A.rowptr[n]);
  for (int64_t p = 0; p < A.rowptr[n]; ++p) scaled[p] = alpha * A.val[p];
  const bool dominant = row_excess(A, dshift, scaled, excess);
  std::vector<std::vector<double>> vupd(dominant ? T.nsup : 0);
  std::vector<int32_t> at;
  int32_t fs = 0;  // first supernode of S in the front
  for (int32_t s = 0; s < T.nsup; ++s) {
    const int32_t f = T.sup_first[s], l = T.sup_first[s + 1];
    const int64_t w = l - f;
    const int32_t* R = &T.sup_rows[T.sup_rowptr[s]];
    const int64_t nr = T.sup_rowptr[s + 1] - T.sup_rowptr[s];
    const int64_t r = nr - w;
    for (int64_t k = 0; k < nr; ++k) pos[R[k]] = (int32_t)k;
    front.assign(nr * nr, 0.0);
    v.assign(nr, 0.0);
    // assemble the columns of diag(dshift) + alpha*A owned by this supernode
    for (int32_t j = f; j < l; ++j) {
      int32_t o = S.perm[j];
      double* colj = &front[(j - f) * nr];
      for (int64_t p = A.rowptr[o]; p < A.rowptr[o + 1]; ++p) {
        int32_t i = S.iperm[A.col[p]];
        if (i < j) continue;
        if (pos[i] < 0) return "row outside the symbolic structure";
        colj[pos[i]] += scaled[p];
      }
      if (dshift) colj[j - f] += dshift[o];
      v[j - f] = excess[o];
    }
    // extend-add the children's update matrices
    for (int32_t c : kids[s]) {
      const int64_t wc = T.sup_first[c + 1] - T.sup_first[c];
      const int32_t* Rc = &T.sup_rows[T.sup_rowptr[c] + wc];
      const int64_t rc = T.sup_rowptr[c + 1] - T.sup_rowptr[c] - wc;
      const std::vector<double>& U = upd[c];
      std::vector<int32_t> rel(rc);
      for (int64_t a = 0; a < rc; ++a) rel[a] = pos[Rc[a]];
      for (int64_t b = 0; b < rc; ++b) {
        double* fc = &front[(int64_t)rel[b] * nr];
        const double* uc = &U[b * rc];
        for (int64_t a = b; a < rc; ++a) fc[rel[a]] += uc[a];
        if (dominant) v[rel[b]] += vupd[c][b];
      }
      std::vector<double>().swap(upd[c]);
    }
    // partial factorisation of the first w columns
    if (!partial_ldlt(front.data(), nr, w, &F.dinv[f], lcol, dominant ? v.data() : nullptr))
      return "matrix is not symmetric positive definite";
    // solve panels of S's supernodes in this front
    for (; fs < S.nsup && S.sup_first[fs] < l; ++fs) {
      const int64_t j0 = S.sup_first[fs] - f, wf = S.sup_first[fs + 1] - S.sup_first[fs];
      const int64_t ld = S.sup_rowptr[fs + 1] - S.sup_rowptr[fs], rf = ld - wf;
      const int32_t* Rf = &S.sup_rows[S.sup_rowptr[fs] + wf];
      at.resize(rf);
      for (int64_t i = 0; i < rf; ++i) at[i] = pos[Rf[i]];
      const int32_t* rows = coarse ? at.data() : nullptr;
      double* pcm = &F.pan_cm[S.pan_off[fs]];
      double* prm = &F.pan_rm[S.pan_off[fs]];
      parallel_for(wf, (double)wf * (double)wf * (double)ld / 2.0, [&](int64_t lo, int64_t hi) {
        for (int64_t k = lo; k < hi; ++k)
          panel_column(front.data(), nr, j0, wf, rf, rows, k, &pcm[k * ld]);
      });
      parallel_for(ld, (double)wf * ld, [&](int64_t lo, int64_t hi) {
        for (int64_t i = lo; i < hi; ++i)
          for (int64_t k = 0; k < wf; ++k) prm[i * wf + k] = pcm[k * ld + i];
      });
    }
    if (coarse_pan) {
      double* pan = &(*coarse_pan)[T.pan_off[s]];
      parallel_for(w, (double)w * (double)w * (double)nr / 2.0, [&](int64_t lo, int64_t hi) {
        for (int64_t k = lo; k < hi; ++k)
          panel_column(front.data(), nr, 0, w, r, nullptr, k, &pan[k * nr]);
      });
    }
    // Schur complement handed to the parent
    if (r > 0 && T.sup_parent[s] >= 0) {
      std::vector<double>& U = upd[s];
      U.assign(r * r, 0.0);
      for (int64_t b = 0; b < r; ++b)
        std::memcpy(&U[b * r + b], &front[(w + b) * nr + w + b], sizeof(double) * (r - b));
      if (dominant) vupd[s].assign(v.begin() + w, v.end());
    }
    for (int64_t k = 0; k < nr; ++k) pos[R[k]] = -1;
  }
  return "";
}

}  // namespace matex
