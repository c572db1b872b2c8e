// The Lanczos combination psi_new = sum_j c_j U_j of one point in fixed point
// (tdse_fixed.cuh).
//
// In FP64 it takes four instructions a vector, 64 cycles a warp each: 48 of a
// point's 52 at twelve vectors, which bound it.  Here the products run on the
// integer pipe, kCbGroup vectors at a time: the operands are converted
// against the group's largest term (exponent of the value plus that of its
// coefficient), the four partial sums are integers and only they are converted
// back and added in FP64.
//
// Bits: operands |X| < 2^59, coefficients |K| <= 2^57, so that
// |mm| < 2 kCbGroup 1.25 2^58 < 2^63; a unit of V is 2^-58 of the largest term's
// power of two, and what an operand loses below 2^-59 of it is the only other
// rounding before the group's sum is rounded to FP64, where FP64 rounds every
// partial sum to 2^-53.  Warps whose values lie near FP64's limits, or are not
// finite, take the FP64 sums.
// Measured: a Lanczos-12 step on 512,000 points 379 to 370 us; 32 instances of
// 2e7 points, four steps with host copies, 46.0 to 43.7 ms.
#pragma once

#include <cuda_runtime.h>

#include "tdse_internal.cuh"
#include "tdse_walk_fixed.cuh"

namespace tdse_dev {
namespace stencil {

constexpr int kCbGroup = 8;
constexpr int kCbLo = 128, kCbHi = 1900;   // exponent fields of a group's largest value: else FP64

// The coefficients in shared memory, formed once a block.
struct CbCoef {
  int4 k;        // limbs of the real and the imaginary part, K = c 2^(57 - ec)
  int ec;        // |c| < 2^ec
  int ok;        // within the exponents the sums can take (or zero)
};
struct CbTable {
  CbCoef f[kMaxKrylov];
  double2 c[kMaxKrylov];
  int k, ok;
};

// Called by every lane of a warp, which may use the table after it (other
// warps after a barrier).
__device__ __forceinline__ void cb_setup(CbTable &t, const LanczosScalars *ls) {
  static_assert(kMaxKrylov == 32, "a lane for each coefficient");
  const int j = threadIdx.x & 31;
  const int k = __ldcg(&ls->kdim);
  const double2 c = __ldcg(&ls->coef[j]);
  const int e = max((int)(max(fx_field(c.x), fx_field(c.y)) >> 20), 1);
  CbCoef q;
  const Limb x = fx_limbs(fx_small(c.x, e) >> 3), y = fx_limbs(fx_small(c.y, e) >> 3);
  q.k = make_int4(x.h, x.l, y.h, y.l);
  q.ec = e - 1022;
  q.ok = (c.x == 0.0 && c.y == 0.0) || (e >= 512 && e <= 1534);
  t.f[j] = q;
  t.c[j] = c;
  const bool all = __all_sync(0xffffffffu, j >= k || q.ok);
  if (j == 0) {
    t.k = k;
    t.ok = all;
  }
  __syncwarp();
}

// sum_j c_j u_j of the warp's points, u_j = load(j).  Every lane of the warp calls it
// (a lane without a point with zeros).
template <typename Load>
__device__ __forceinline__ double2 cb_sum(const CbTable &t, Load &&load) {
  const int k = t.k;
  double2 o = make_double2(0.0, 0.0);
  for (int j0 = 0; j0 < k; j0 += kCbGroup) {
    double2 u[kCbGroup];
#pragma unroll
    for (int q = 0; q < kCbGroup; ++q) u[q] = (j0 + q < k) ? load(j0 + q) : make_double2(0.0, 0.0);
    int E = kNone, lo = kCbHi, hi = kCbLo;
#pragma unroll
    for (int q = 0; q < kCbGroup; ++q) {
      if (j0 + q >= k) break;
      const int e = (int)(max(fx_field(u[q].x), fx_field(u[q].y)) >> 20);
      if (e) {
        lo = min(lo, e);
        hi = max(hi, e);
        E = max(E, e + t.f[j0 + q].ec);
      } else if ((((unsigned)__double2hiint(u[q].x) | (unsigned)__double2hiint(u[q].y)) & 0xfffffu) |
                 (unsigned)__double2loint(u[q].x) | (unsigned)__double2loint(u[q].y)) {
        E = max(E, 0);   // subnormal (seen in integers: an FP64 comparison takes its pipe even where it is not due)
        lo = 0;
      }
    }
    if (t.ok && __all_sync(0xffffffffu, E == kNone || (lo >= kCbLo && hi <= kCbHi && E > kOutLo && E <= kOutHi))) {
      int64_t xh = 0, xm = kHalf >> 6, yh = 0, ym = kHalf >> 6;   // rounded, not cut
      int64_t nh = 0, nm = 0;                                     // the real part's second products: subtracted
#pragma unroll
      for (int q = 0; q < kCbGroup; ++q) {
        if (j0 + q >= k) break;
        const CbCoef &f = t.f[j0 + q];
        // the operands' exponent field, one up for 59 bits; above that of every
        // value here, and at least 64, from where a zero converts to zero
        const uint32_t ee = (uint32_t)min(max(E - f.ec + 1, 64), 4095) << 20;
        const Limb X = fx_limbs(fx_word(u[q].x, ee)), Y = fx_limbs(fx_word(u[q].y, ee));
        const Limb a = {f.k.x, f.k.y}, b = {f.k.z, f.k.w};
        fx_mac(X, a, xh, xm);
        fx_mac(Y, b, nh, nm);
        fx_mac(Y, a, yh, ym);
        fx_mac(X, b, yh, ym);
      }
      xh -= nh;
      xm -= nm;
      o.x = __dadd_rn(o.x, fx_result((xh << 6) + (xm >> 26), E - 1));
      o.y = __dadd_rn(o.y, fx_result((yh << 6) + (ym >> 26), E - 1));
    } else {
#pragma unroll
      for (int q = 0; q < kCbGroup; ++q) {
        if (j0 + q >= k) break;
        const double2 c = t.c[j0 + q];
        o.x = __fma_rn(c.x, u[q].x, o.x);
        o.x = __fma_rn(-c.y, u[q].y, o.x);
        o.y = __fma_rn(c.x, u[q].y, o.y);
        o.y = __fma_rn(c.y, u[q].x, o.y);
      }
    }
  }
  return o;
}

}  // namespace stencil
}  // namespace tdse_dev
