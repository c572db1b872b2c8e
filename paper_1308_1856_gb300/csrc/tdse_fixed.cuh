// Fixed-point arithmetic for the FP64 stencil: 60-bit integers that share a
// block's exponent, multiplied and summed on the integer pipe.
//
// Why: on GB300 an FP64 instruction of a warp holds its SM sub-partition's
// FP64 pipe for 64 cycles, a 32 x 32 + 64-bit integer multiply-add 2 cycles
// (both measured).  H x takes 15 FP64 instructions a point, 960 cycles a warp;
// the same sums as integer limb products take about a third of that, and they
// leave the FP64 pipe to the epilogue.
//
// Representation.  A block of doubles (in the stencil: the two parts of one value)
// with largest exponent field e holds each as a 60-bit two's complement integer X,
//   x = X 2^(e - 1082),  |X| < 2^60,
// so the block's largest values keep 7 bits more than a double's 53 and any
// value down to 2^-7 of the largest is exact.  A coefficient is held against an
// exponent ec of its own, c = K 2^(ec - 61), |K| <= 2^61.  Products are formed
// from 32-bit limbs, X = xh 2^32 + xl with xl signed:
//   X K = xh kh 2^64 + (xh kl + xl kh) 2^32 + xl kl.
// hh and mm below are the first two sums over all terms of a point, each operand
// shifted to the exponent T - ec of the sum first (T: the largest of the terms' e +
// ec); the last (below 2^62) is dropped, and V = (hh 2^64 + mm 2^32) / 2^61 is
// rounded.  One unit u of V is 2^(T - 1082).
//
// Error.  The dropped products of the five terms are below 2 u each, the cuts of
// the operands (in the conversion and in the shift) and of the coefficients below 12 u
// together: V is off by less than 24 u, typically by 2 u.  The largest of a point's
// own terms is at least 2^(T - 1027) (fx_scale, fx_stencil_coef and the walker's
// kDiagHigh see to that), 2^55 u, so that the worst case is 6 2^-53 of the terms'
// sum in modulus.  FP64 rounds six partial sums and reaches the same.
//
// Sums fit: with five products (stencil sums up to 2^61 with coefficients up to
// 2^59, the diagonal's to 2^61, the couplings' to 2^61 / 3^(1/2)) |mm| < 6.2 2^60 and
// |hh| < 2^59; the velocity gauge's two more (operands of 58 bits) make it 7.6 2^60.
//
// The functions are plain C on integers, compiled for the host as well, where
// they are tested against 128-bit arithmetic.
#pragma once

#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace tdse_fx {

constexpr uint32_t kExpMask = 0x7ff00000u;   // exponent field of a double's high word
// Block exponents from here on convert by fx_from_words, where a zero beside
// the block's largest value comes out as zero; smaller ones by fx_from_small.
constexpr int kExpSmall = 64;
// Exponents (E of fx_to_bits) that give a normal double for any V != 0.
constexpr int kOutLo = 64, kOutHi = 2000;
constexpr int kNone = -(1 << 24);            // "no term": below every exponent, far enough to subtract from
constexpr int kDiagBits = 5;                 // low bits of an encoded diagonal entry: its own shift
constexpr int kDiagMask = (1 << kDiagBits) - 1;

struct Limb {
  int h, l;   // X = h 2^32 + l
};

// The limbs of a 64-bit integer: l is the low word read as signed, h takes the carry.
FX_HD Limb fx_limbs(int64_t X) {
  Limb r;
  const uint32_t lo = (uint32_t)(uint64_t)X, hi = (uint32_t)((uint64_t)X >> 32);
  r.l = (int)lo;
#ifdef __CUDA_ARCH__
  // lo >> 31 as the carry of lo + 2^31: two adds (1 cycle each) instead of a shift (2) and an add
  asm("{\n .reg .u32 t;\n add.cc.u32 t, %1, 0x80000000;\n addc.u32 %0, %2, 0;\n}" : "=r"(r.h) : "r"(lo), "r"(hi));
#else
  r.h = (int)(hi + (lo >> 31));
#endif
  return r;
}

FX_HD int64_t fx_signed(uint64_t mag, uint32_t hi) {   // mag with the sign bit of hi
#ifdef __CUDA_ARCH__
  int64_t X = (int64_t)mag;
  asm("{\n .reg .pred p;\n setp.lt.s32 p, %1, 0;\n @p neg.s64 %0, %0;\n}" : "+l"(X) : "r"(hi));
  return X;
#else
  return (int32_t)hi < 0 ? -(int64_t)mag : (int64_t)mag;
#endif
}

// A double (its two words) against the block's largest exponent field emax
// (in place, as in the high word; >= this value's).
FX_HD int64_t fx_from_words(uint32_t hi, uint32_t lo, uint32_t emax) {
  const uint64_t M = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const uint32_t d = (emax - (hi & kExpMask)) >> 20;
  const uint32_t n = d + 3u < 63u ? d + 3u : 63u;
  return fx_signed((M << 10) >> n, hi);
}

// The same for a block whose largest exponent field is small: e = max(1, that
// field), zeros and subnormal values exact.
FX_HD int64_t fx_from_small(uint32_t hi, uint32_t lo, int e) {
  const int f = (int)((hi & kExpMask) >> 20);
  const uint64_t M = ((uint64_t)((hi & 0xfffffu) | (f ? 0x100000u : 0u)) << 32) | lo;
  const int d = e - (f ? f : 1);
  const int n = d + 3 < 63 ? d + 3 : 63;
  return fx_signed((M << 10) >> n, hi);
}

// a b + c, one instruction (the accumulator's start value needs no move)
FX_HD int64_t fx_mad(int a, int b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return c + (int64_t)a * b;
#endif
}
FX_HD void fx_mac(const Limb &x, const Limb &k, int64_t &hh, int64_t &mm) {
  hh = fx_mad(x.h, k.h, hh);
  mm = fx_mad(x.h, k.l, mm);
  mm = fx_mad(x.l, k.h, mm);
}

constexpr int64_t kHalf = (int64_t)1 << 31;   // mm's start value: V is rounded, not cut

// V = (hh 2^64 + mm 2^32) 2^(bits - 64), mm started at kHalf >> bits.
FX_HD int64_t fx_value(int64_t hh, int64_t mm, int bits = 0) {
  return (int64_t)((uint64_t)hh << bits) + (mm >> (32 - bits));
}
constexpr int kFineBits = 3;   // of the walker, whose sums stay below 7 2^56 without them

// The product of two coefficients as a coefficient: K1 K2 / 2^60 (K1 against 2^0
// is kappa 2^61, K2 an operand-format value below 2^60).
FX_HD int64_t fx_coef_product(const Limb &a, const Limb &b) {
  int64_t hh = 0, mm = 0;
  fx_mac(a, b, hh, mm);
  return (int64_t)((uint64_t)hh << 4) + (mm >> 28);
}

FX_HD int fx_clz(uint64_t a) {
#ifdef __CUDA_ARCH__
  const uint32_t h = (uint32_t)(a >> 32);
  return h ? __clz(h) : 32 + __clz((uint32_t)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// The bits of the double V 2^(E - 1079), rounded to nearest; E in [kOutLo, kOutHi].
FX_HD uint64_t fx_to_bits(int64_t V, int E) {
  const uint64_t sign = (uint64_t)V & 0x8000000000000000ull;
  const uint64_t A = V < 0 ? (uint64_t)-V : (uint64_t)V;
  const int lz = fx_clz(A);
  const uint64_t m = A << lz;
  // the leading one of the mantissa adds one to the exponent field
  const uint64_t f = (uint64_t)(uint32_t)(E + 6 - lz) << 52;
  const uint64_t b = sign | (f + (m >> 11) + ((m >> 10) & 1u));
  return A ? b : 0;
}

// The leading zeros of the larger of two values, less the six above 58 bits ...
FX_HD int fx_lead(int64_t a, int64_t b) {
  return fx_clz((uint64_t)(a < 0 ? -a : a) | (uint64_t)(b < 0 ? -b : b)) - 6;
}
// ... and a value brought to 58 bits by them.
FX_HD int64_t fx_bring(int64_t v, int n) { return n < 0 ? v >> -n : (int64_t)((uint64_t)v << n); }

// A warp's sum of 32 doubles: each is held as a 58-bit integer against the
// largest exponent field e of the warp (kSumLo <= e <= kSumHi), rounded to
// nearest, v = X 2^(e - kSumBias), |X| <= 2^57, so that the sum stays below 2^62;
// the values within 2^-4 of the largest are exact and the others are off by at
// most half of 2^-57 of the largest's power of two, where an FP64 addition rounds
// to 2^-53 of its sum.  The integers are added as three pieces of 20, 20 and 18 bits.
constexpr int kSumBias = 1079, kSumLo = 128, kSumHi = 2000;
FX_HD int64_t fx_addend(uint32_t hi, uint32_t lo, int e) {
  const int f = (int)((hi & kExpMask) >> 20);
  const uint64_t M = ((uint64_t)((hi & 0xfffffu) | (f ? 0x100000u : 0u)) << 32) | lo;
  const int d = e - f;                                 // subnormal values (f = 0) fall below the last bit
  return fx_signed((((M << 5) >> (d < 63 ? d : 63)) + 1) >> 1, hi);
}
FX_HD int64_t fx_total(uint32_t p0, uint32_t p1, int32_t p2) {
  return (int64_t)(((uint64_t)(int64_t)p2 << 40) + ((uint64_t)p1 << 20) + p0);
}

// sqrt(s2) and its inverse from y, a few units in the last place off 1 / sqrt(s2):
// one Newton step each on an exactly formed residual (P. Markstein, IBM J. Res.
// Dev. 34 (1990) 111), within 0.51 of a unit as a square root and a division, each
// rounded, are within 1.
FX_HD void fx_norm(double s2, double y, double &nrm, double &inv) {
  const double g = s2 * y;
  nrm = fma(0.5 * y, fma(-g, g, s2), g);
  inv = fma(y, fma(-nrm, y, 1.0), y);
}

// A neighbour's coefficient c = q 2^(e - 61), 2^58 <= |q| < 2^59: exact.
struct FxStencilCoef {
  int64_t q;
  int e;
};
inline FxStencilCoef fx_stencil_coef(double c) {
  FxStencilCoef r = {0, kNone};
  if (c == 0.0) return r;
  int e = 0;
  const double m = frexp(c, &e);          // |m| in [1/2, 1)
  r.q = (int64_t)(m * 576460752303423488.0);   // 2^59
  r.e = e + 2;
  return r;
}

// The exponent of the diagonal's coefficients: room for
// diagonal entries of more than twice c0, the value the diagonal tends to;
// larger ones (the centrifugal term next to the origin) carry a shift of their
// own.  false: a grid spacing outside 2^+-30, left to the FP64 path.
FX_HD bool fx_scale(double c0, int &ec) {
  if (!(c0 > 8.7e-19 && c0 < 1.1e18)) return false;   // 2^-60 .. 2^60
  int e = -62;
  for (double p = 2.168404344971009e-19; p <= c0; p *= 2.0) ++e;   // p = 2^e: the loop ends with 2^e > c0
  ec = e + 2;
  return true;
}

// A diagonal entry D = m 2^(ec + s - 61): m with s in its low kDiagBits bits
// (zero in m: for |D| near c0 those bits lie below a double's last one).
// |D| < 2^(ec + kDiagMask) is the caller's to check (fx_diag_fits).
FX_HD int64_t fx_encode_diag(uint64_t bits, int ec) {
  const int F = (int)((bits >> 52) & 0x7ff);
  if (F == 0) return 0;
  const uint64_t M = (bits & 0xfffffffffffffull) | 0x10000000000000ull;
  const int s = F - 1022 > ec ? F - 1022 - ec : 0;
  const int t = F - 1019 - ec - s;        // |D| = M 2^(F - 1075); units of 2^(ec + s - 56)
  uint64_t q = 0;
  if (t >= 0) q = M << t;                 // t <= 3
  else if (t > -60) q = (M + (1ull << (-t - 1))) >> -t;
  const int64_t m = (int64_t)(q << kDiagBits);
  return ((bits >> 63) ? -m : m) + s;
}
inline bool fx_diag_fits(double bound, int ec) {
  double lim = 1.0;
  for (int k = 0; k < (ec < 0 ? -ec : ec); ++k) lim *= ec < 0 ? 0.5 : 2.0;
  return bound < lim * 1073741824.0;      // 2^(ec + 30): false for NaN too
}

FX_HD int64_t fx_diag_value(int64_t q) { return q & ~(int64_t)kDiagMask; }
FX_HD int fx_diag_shift(int64_t q) { return (int)(q & kDiagMask); }

// K = c 2^(61 - ec) of a coefficient with |c| < 2^ec, cut below its 60 bits.
FX_HD int64_t fx_coef(uint64_t bits, int ec) {
  return 2 * fx_from_words((uint32_t)(bits >> 32), (uint32_t)bits, (uint32_t)(ec + 1022) << 20);
}

}  // namespace tdse_fx
