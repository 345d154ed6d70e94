// Split of FP64 values into seven signed 8-bit digits, for products on the FP16
// tensor cores that are as accurate as FP64 relative to the largest entries that
// meet (digits, products and sums are exact, the 55-bit operands rounded; the
// Ozaki scheme:
// Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59, 2012).
//
// A row (column) whose largest entry is below 1.984 2^(e - 1023) is scaled to the
// integers q = round(v 2^(1077 - e)), |q| < 127 2^48 (e is that entry's biased
// exponent, or one more where its mantissa is 1.984 and up), and
// q + sum_p 128 256^p is cut into its seven bytes u_p: the digits u_p - 128 lie
// in [-128, 127] (the leading one in [-127, 127]) and are exact in FP16.  One
// split keeps 55 bits below the largest entry.  With digit 0 the leading one, the
// products of digits with p + r = d <= 6 go to the FP32 accumulator d: at most
// 7 2^14 128 < 2^24 over 128 reduction values, an exact integer in whatever order
// the tensor core adds.  The six products with p + r = 7 join accumulator 6 as
// a_p 2^-8: what FP32 rounds off there is below 2^-60 of max|row| max|column|,
// what is left out (p + r > 7) below 2^-61 a term; without those six the left-out
// part is as large as an FP64 dot product's rounding.  The sum is kept in units of
// 2^-54 of the two maxima's powers of two: a lone term of two small mantissas is
// off by 2^-53 of itself at most.  What remains is the rounding of the operands, by
// the same amount for large and small entries: solutions of the grids' two
// matrices (576 to 57,600 nodes, one to four layers) are off by 0.29e-15 to
// 0.58e-15 in the root mean square, by 0.23e-15 to 0.36e-15 with the FP64 kernels on
// the same factors.  (One bit less in either operand, with the leading digit in
// [-64, 64], and the sum in units of 2^-52: 0.6e-15 to 1.2e-15.)
// The FP64 pipe, 16 clocks per warp instruction and SM on GB300 (measured), is
// left one conversion per result; the split runs on the integer pipe.
#pragma once
#include <cstdint>

namespace matex {
namespace s8 {

constexpr int kDigits = 7;
constexpr int kChunkSteps = 8;               // K steps (of 16) one exact sum may cover
// Panel tile, 8 rows x 16 terms, mma.sync's B operand: per lane digits 0..3,
// 4..5 and 6 of its four terms (a byte each), the rows' exponents (int16), the
// nodes their results go to (int32).
constexpr int kTile45 = 512, kTile6 = 768, kTileE = 896, kTileDst = kTileE + 16,
              kTileBytes = kTileDst + 32;
constexpr int kFragBytes = kDigits * 512;    // 16 right-hand sides x 16 terms, the A operand, FP16
constexpr uint64_t kBias = 0x0080808080808080ull;
constexpr int kNonFinite = 1 << 20;          // exponent mark of a column with an inf or NaN
constexpr float kBiasedZero = 12582912.f;    // 1.5 2^23: sums below 2^22 sit in the mantissa
constexpr int kKeyInf = 0x7ff04000;          // key of an inf; a NaN's is that or larger

// largest-exponent key of a value: its high word without the sign, mantissas from
// 1.984 on carried into the next exponent
__device__ __forceinline__ int exp_key(double v) {
  return min(__double2hiint(v) & 0x7fffffff, 0x7ff80000) + 0x4000;
}
__device__ __forceinline__ int key_exp(int key) { return max(key >> 20, 1); }

// The biased digits of v on the scale of exponent e, at least its key's (bytes
// 0..6, leading digit in byte 6).
__device__ __forceinline__ uint64_t digits(double v, int e) {
  const int hi = __double2hiint(v);
  const int ev = (hi >> 20) & 0x7ff;
  const uint32_t mh = (hi & 0xfffff) | (ev ? 0x100000u : 0u);
  const uint64_t m8 = (((uint64_t)mh << 32) | (uint32_t)__double2loint(v)) << 3;
  const int sh = min(e - max(ev, 1), 63);
  uint64_t q = ((m8 >> sh) + 1) >> 1;  // rounded to nearest
  if (hi < 0) q = 0 - q;
  return q + kBias;
}

// bytes (0, 1) or (2, 3) of x as two FP16 integers byte - 128: the byte is
// the low mantissa of 1024 + byte
template <int kHalf>
__device__ __forceinline__ uint32_t widen(uint32_t x) {
  uint32_t y = __byte_perm(x, 0x64646464u, kHalf ? 0x4342 : 0x4140);
  asm("sub.f16x2 %0, %0, %1;" : "+r"(y) : "r"(0x64806480u));
  return y;
}

// FP16 digits of the value pair (x, y): out[d] holds digit d of both
__device__ __forceinline__ void widen_pair(uint64_t x, uint64_t y, uint32_t (&out)[kDigits]) {
  const uint32_t xl = (uint32_t)x, xh = (uint32_t)(x >> 32), yl = (uint32_t)y,
                 yh = (uint32_t)(y >> 32);
  const uint32_t t0 = __byte_perm(xl, yl, 0x5140), t1 = __byte_perm(xl, yl, 0x7362);
  const uint32_t t2 = __byte_perm(xh, yh, 0x5140), t3 = __byte_perm(xh, yh, 0x7362);
  out[6] = widen<0>(t0);
  out[5] = widen<1>(t0);
  out[4] = widen<0>(t1);
  out[3] = widen<1>(t1);
  out[2] = widen<0>(t2);
  out[1] = widen<1>(t2);
  out[0] = widen<0>(t3);
}

// two FP16 integers times 2^-8 (exact)
__device__ __forceinline__ uint32_t down8(uint32_t x) {
  uint32_t y;
  asm("mul.f16x2 %0, %1, %2;" : "=r"(y) : "r"(x), "r"(0x1C001C00u));
  return y;
}

// D += A B, m16n8k16, FP16 digits, FP32 sums c[.][d] (mma.sync's four results)
__device__ __forceinline__ void mma(float (&c)[4][kDigits], int d, const uint4& a, uint32_t b0,
                                    uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0][d]), "+f"(c[1][d]), "+f"(c[2][d]), "+f"(c[3][d])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// rare results: subnormal, overflow, a column that held an inf or NaN
static __device__ __noinline__ double compose_slow(long long s, int e) {
  if (e >= kNonFinite / 2) return __longlong_as_double(0x7ff8000000000000ll);
  return s == 0 ? 0.0 : ldexp((double)s, e - 2098);
}

// The FP64 value of the seven sums c_d (d = p + r) with row and column
// exponents adding to e: S 2^(e - 2098), S = sum_d c_d 2^(8 (5 - d)), the last
// sum rounded to that unit.  |S| < 2^62 is rounded once, by the conversion;
// the power of two is added to the exponent field.  The sums of d < 2 stay
// below 2^22 over a whole chunk and carry kBiasedZero; with kFew (at most two
// K steps) all do.
template <bool kFew>
__device__ __forceinline__ double compose(const float (&c)[kDigits], int e) {
  int v[kDigits];
#pragma unroll
  for (int d = 0; d < kDigits; ++d)
    v[d] = kFew || d < 2 ? __float_as_int(c[d]) - __float_as_int(kBiasedZero) : __float2int_rn(c[d]);
  long long s = (long long)v[4] * 256 + (v[5] + ((v[6] + 128) >> 8));
  s += (long long)v[3] * 65536;
  s += (long long)(v[1] * 256 + v[2]) * 16777216;
  s += (long long)v[0] << 40;
  // exponent fields of (double)s: 1023 .. 1085; zeros (padded rows, unloaded
  // nodes) are common and stay out of the call
  const bool zero = s == 0 && e < kNonFinite / 2;
  if (!zero && (unsigned)(e - 1076) > 1982u) return compose_slow(s, e);
  const double x = (double)s;
  return zero ? 0.0 : __hiloint2double(__double2hiint(x) + (e - 2098) * (1 << 20), __double2loint(x));
}

}  // namespace s8
}  // namespace matex
