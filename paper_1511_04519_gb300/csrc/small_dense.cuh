// Small dense linear algebra on m x m matrices in shared memory with leading
// dimension LD, executed cooperatively by a thread group (a CTA, a part of one
// or one warp: the template parameter G): products, a pivoted Gaussian solve,
// the matrix exponential by scaling and squaring with the degree-19 Taylor
// polynomial, and the rational Hessenberg map of Eq. 9.  Used for e^{h H_m}
// (LD = 20) and for Frechet derivatives through the 2m x 2m block exponential
// (LD = 40).
//
// What bounds them: an FP64 instruction of a warp takes 66 clocks, issued alone
// or in a chain, whatever its active lanes, a division 650 (measured on GB300).
// Hence the Taylor polynomial (seven products, 20 multiply-adds beside them and
// no division, where a [13/13] Pade approximant has six products and a Gaussian
// solve of 2m divisions), the norm by integer operations, one division per pivot,
// and independent exponentials on separate groups of warps.
#pragma once
#include "kernels.h"

namespace matex {

constexpr int kSmallThreads = 128;
// threads of the batched residual and coefficient kernels: three exponentials
// at once, 64 threads each (64 entries of a matrix per pass)
constexpr int kWorkThreads = 64, kTeamThreads = 192;

// 1 / k!, k = 0..19: the degree-19 Taylor polynomial of e^x is within
// 1.06 / 20! < 5e-19 of e^x for |x| <= 1.
constexpr int kTaylorDeg = 19;
struct InvFactorials {
  double c[kTaylorDeg + 1];
};
__host__ __device__ constexpr InvFactorials inv_factorials() {
  InvFactorials r{};
  double f = 1.0;  // 19! < 2^57 carries no rounding up to 18!, one at 19!
  for (int k = 0; k <= kTaylorDeg; ++k) {
    if (k > 0) f *= (double)k;
    r.c[k] = 1.0 / f;
  }
  return r;
}

// Work arrays of one exponential (shared memory)
template <int LD>
struct SmallWork {
  double A[LD * LD], A2[LD * LD], A3[LD * LD], A4[LD * LD], A5[LD * LD], V[LD * LD], T[LD * LD];
  double inv[LD];  // reciprocal pivots
  int key[LD];     // column norms, as exponents
  int piv;
};

// The threads that run the routines below together: a whole CTA, 64 threads of
// one, or one warp (the others do not take part and must not touch the work
// arrays).
struct CtaGroup {
  static __device__ __forceinline__ int rank() { return threadIdx.x; }
  static __device__ __forceinline__ int size() { return blockDim.x; }
  static __device__ __forceinline__ void sync() { __syncthreads(); }
};
struct WorkGroup {  // threads 64 w .. 64 w + 63, named barrier 1 + w
  static __device__ __forceinline__ int rank() { return threadIdx.x % kWorkThreads; }
  static __device__ __forceinline__ int size() { return kWorkThreads; }
  static __device__ __forceinline__ void sync() {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / kWorkThreads), "n"(kWorkThreads)
                 : "memory");
  }
};
struct WarpGroup {
  static __device__ __forceinline__ int rank() { return threadIdx.x & 31; }
  static __device__ __forceinline__ int size() { return 32; }
  static __device__ __forceinline__ void sync() { __syncwarp(); }
};

template <int LD, class G = CtaGroup>
struct Small {
  static constexpr int kLd = LD;
  static constexpr int kMat = LD * LD;
  using Work = SmallWork<LD>;
  static __device__ void mat_mul(const double* A, const double* B, double* C, int m) {
  for (int e = G::rank(); e < m * m; e += G::size()) {
    const int i = e / m, j = e - i * m;
    double s = 0.0;
    for (int k = 0; k < m; ++k) s = fma(A[i * kLd + k], B[k * kLd + j], s);
    C[i * kLd + j] = s;
  }
  G::sync();
}

// Solve Q X = P in place (X overwrites P), Gaussian elimination with partial
// pivoting; Q is destroyed.  One division per pivot, kept in inv.  Sizes of
// entries are compared as bit patterns (integers; a NaN counts as largest).
  static __device__ void lu_solve(double* Q, double* P, int m, int* piv_sh, double* inv) {
  auto size_key = [](double v) { return __double_as_longlong(v) & 0x7fffffffffffffffll; };
  for (int k = 0; k < m; ++k) {
    if (G::rank() == 0) {
      int p = k;
      long long best = size_key(Q[k * kLd + k]);
      for (int i = k + 1; i < m; ++i) {
        const long long a = size_key(Q[i * kLd + k]);
        if (a > best) { best = a; p = i; }
      }
      *piv_sh = p;
      inv[k] = 1.0 / Q[p * kLd + k];
    }
    G::sync();
    const int p = *piv_sh;
    if (p != k) {
      for (int c = G::rank(); c < m; c += G::size()) {
        double t = Q[k * kLd + c]; Q[k * kLd + c] = Q[p * kLd + c]; Q[p * kLd + c] = t;
        t = P[k * kLd + c]; P[k * kLd + c] = P[p * kLd + c]; P[p * kLd + c] = t;
      }
      G::sync();
    }
    const double iv = inv[k];
    const int rows = m - k - 1, cols = 2 * m - k - 1;  // Q's columns right of k, P's
    for (int e = G::rank(); e < rows * cols; e += G::size()) {
      const int i = k + 1 + e / cols, c = e % cols;
      const double f = Q[i * kLd + k] * iv;  // column k itself is not read again below row k
      double* row = c < m - k - 1 ? Q + k + 1 + c : P + c - (m - k - 1);
      row[i * kLd] = fma(-f, row[k * kLd], row[i * kLd]);
    }
    G::sync();
  }
  // back substitution, one thread per right-hand-side column
  for (int c = G::rank(); c < m; c += G::size()) {
    for (int k = m - 1; k >= 0; --k) {
      double s = P[k * kLd + c];
      for (int i = k + 1; i < m; ++i) s = fma(-Q[k * kLd + i], P[i * kLd + c], s);
      P[k * kLd + c] = s * inv[k];
    }
  }
  G::sync();
}

// The smallest s >= 0 with ||A||_1 2^-s <= 1, from the columns' sums taken on
// 24 bits rounded up (integers and FP32; an inf or NaN entry: s = 1026).
  static __device__ int scale_steps(const double* A, int m, int* key) {
  for (int j = G::rank(); j < m; j += G::size()) {
    int top = 0;  // largest biased exponent of the column
    for (int i = 0; i < m; ++i) top = max(top, (__double2hiint(A[i * kLd + j]) >> 20) & 0x7ff);
    float f = 0.f;
    for (int i = 0; i < m; ++i) {
      const double v = A[i * kLd + j];
      const int hi = __double2hiint(v), d = top - ((hi >> 20) & 0x7ff);
      const int mant = ((hi & 0xfffff) << 3) | ((unsigned)__double2loint(v) >> 29);
      if (d < 40) f += __int_as_float(((127 - d) << 23) | mant) * 1.000001f;
    }
    // f 2^(top - 1023) bounds the column's sum: f in [1, 2m)
    const int fe = (__float_as_int(f) >> 23) - 127;
    key[j] = top == 0 ? -2000 : top - 1023 + fe + ((__float_as_int(f) & 0x7fffff) != 0 ? 1 : 0);
  }
  G::sync();
  int e = 0;
  for (int j = 0; j < m; ++j) e = max(e, key[j]);
  G::sync();
  return min(e, 1026);
}

// E = expm(h * M) by scaling and squaring: A = 2^-s h M with norm <= 1, the
// degree-19 Taylor polynomial as four blocks of five terms in powers of A^5
// (Paterson and Stockmeyer 1973), s squarings.  The first two squarings work on
// X = E - I (X -> X^2 + 2 X), where the slow modes keep their relative accuracy
// while no mode has decayed below e^-4: the error is then below that of the
// [13/13] Pade approximant with its 2.4 squarings fewer (root mean square over
// 200 matrices each: 0.4 to 0.8 of it on random Hessenberg matrices of 1 to 20
// rows, 0.5 to 0.7 on stiff Arnoldi ones; squaring E alone 0.7 to 2.2).  M and E
// may not alias work arrays; E may alias M.
  static __device__ void expm(const double* M, double h, double* E, int m, Work& w) {
  constexpr InvFactorials inv = inv_factorials();
  for (int e = G::rank(); e < m * m; e += G::size()) {
    const int i = e / m, j = e - i * m;
    w.A[i * kLd + j] = h * M[i * kLd + j];
  }
  G::sync();
  const int steps = scale_steps(w.A, m, w.key);
  if (steps > 0) {
    const double sc = ldexp(1.0, -steps);
    for (int e = G::rank(); e < m * m; e += G::size()) {
      const int i = e / m, j = e - i * m;
      w.A[i * kLd + j] *= sc;
    }
    G::sync();
  }
  mat_mul(w.A, w.A, w.A2, m);
  for (int e = G::rank(); e < 2 * m * m; e += G::size()) {  // A^3 and A^4
    const int half = e >= m * m ? 1 : 0, x = e - half * m * m, i = x / m, j = x - i * m;
    const double* L = half ? w.A2 : w.A;
    double s = 0.0;
    for (int k = 0; k < m; ++k) s = fma(L[i * kLd + k], w.A2[k * kLd + j], s);
    (half ? w.A4 : w.A3)[i * kLd + j] = s;
  }
  G::sync();
  mat_mul(w.A2, w.A3, w.A5, m);
  double *cur = w.V, *nxt = w.T;
#pragma unroll
  for (int b = 3; b >= 0; --b) {
    for (int e = G::rank(); e < m * m; e += G::size()) {
      const int i = e / m, j = e - i * m, x = i * kLd + j;
      double s = inv.c[5 * b + 4] * w.A4[x];
      s = fma(inv.c[5 * b + 3], w.A3[x], s);
      s = fma(inv.c[5 * b + 2], w.A2[x], s);
      s = fma(inv.c[5 * b + 1], w.A[x], s);
      if (b < 3)
        for (int k = 0; k < m; ++k) s = fma(cur[i * kLd + k], w.A5[k * kLd + j], s);
      if (i == j && b > 0) s += inv.c[5 * b];
      (b < 3 ? nxt : cur)[x] = s;
    }
    G::sync();
    if (b < 3) {
      double* t = cur; cur = nxt; nxt = t;
    }
  }
  const int shifted = min(steps, 2);
  for (int k = 0; k < steps; ++k) {
    if (k < shifted) {
      for (int e = G::rank(); e < m * m; e += G::size()) {
        const int i = e / m, j = e - i * m;
        const double x = cur[i * kLd + j];
        double s = x + x;
        for (int l = 0; l < m; ++l) s = fma(cur[i * kLd + l], cur[l * kLd + j], s);
        if (k + 1 == shifted && i == j) s += 1.0;
        nxt[i * kLd + j] = s;
      }
      G::sync();
    } else {
      mat_mul(cur, cur, nxt, m);
    }
    double* t = cur; cur = nxt; nxt = t;
  }
  for (int e = G::rank(); e < m * m; e += G::size()) {
    const int i = e / m, j = e - i * m;
    E[i * kLd + j] = steps == 0 && i == j ? cur[i * kLd + j] + 1.0 : cur[i * kLd + j];
  }
  G::sync();
}

// The exponent matrix of the Krylov space from its Arnoldi Hessenberg Ht (the
// column's kMaxB x kMaxM array): variant 0 rational, H = (I - Ht_m^{-1}) / gamma
// (Eq. 9); 1 inverted, H = -Ht_m^{-1} (the Arnoldi of G^{-1} C = -A^{-1},
// Sec. 3.3.1); 2 standard, H = Ht_m (the Arnoldi of A, Sec. 2.3).
  static __device__ void rational_H(const double* Ht, int m, double gamma, double* H, Work& w,
                                    int variant = 0) {
  if (variant == 2) {
    for (int e = G::rank(); e < m * m; e += G::size()) {
      const int i = e / m, j = e - i * m;
      H[i * kLd + j] = Ht[i * kMaxM + j];
    }
    G::sync();
    return;
  }
  for (int e = G::rank(); e < m * m; e += G::size()) {
    const int i = e / m, j = e - i * m;
    w.V[i * kLd + j] = Ht[i * kMaxM + j];
    w.T[i * kLd + j] = (i == j) ? 1.0 : 0.0;
  }
  G::sync();
  lu_solve(w.V, w.T, m, &w.piv, w.inv);  // T = Ht_m^{-1}
  if (variant == 1) {
    for (int e = G::rank(); e < m * m; e += G::size()) {
      const int i = e / m, j = e - i * m;
      H[i * kLd + j] = -w.T[i * kLd + j];
    }
  } else {
    const double ig = 1.0 / gamma;
    for (int e = G::rank(); e < m * m; e += G::size()) {
      const int i = e / m, j = e - i * m;
      H[i * kLd + j] = ((i == j ? 1.0 : 0.0) - w.T[i * kLd + j]) * ig;
    }
  }
  G::sync();
}

};

}  // namespace matex
