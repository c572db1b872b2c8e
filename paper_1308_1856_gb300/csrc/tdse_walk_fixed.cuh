// The FP64 operator's row walker in fixed point (tdse_fixed.cuh): H x of either
// gauge with the operand and the result in FP64.
//
// A warp owns a strip of kFxCols radial columns and walks it up the partial
// waves.  Lane k holds columns j0 - 2 + 2k and the one after it, so lanes 0
// and 31 carry the stencil's halo and lanes 1..30 produce results: 60 of 64
// columns useful, every operand value loaded and converted once per strip, the
// radial neighbours exchanged by shuffles.  Two columns a lane halve the
// shuffles and the row's uniform work against one, and take 94% of the lanes'
// work against 88% for the same halo.
//
// Exponents are local to a point: a column is converted against its own exponent,
// and a point's sum is formed against the largest of its own terms', each operand
// shifted there by itself.  What FP64 keeps at a small value beside large ones,
// next to the origin in a high partial wave, inside a wall or among scattered values, is
// kept here too: over such states and ordinary ones the error at a point is at most
// 4.6 2^-53 of its terms' sum in modulus, 0.1 to 0.9 2^-53 in the mean square, where the
// FP64 walk has 5.8 and 0.3 to 1.1 2^-53, in each of them more in the mean square.  One
// exponent for the lane's two columns and their neighbours, six in all, was 1 to 8%
// faster (velocity gauge 5 to 13%: H x of 512,000 points 17.4 us, 19.7 now) but
// lost up to every digit there.
//
// The velocity gauge couples the rows l -+ 1 through their first derivatives and
// l/r terms: four products a part in place of two, of the derivative's integer
// difference D and of the values, and the parts cross (-i).  D of a row is formed
// once, when the row is converted, and kept in the lane's shared memory until
// the row after next, in 58 bits of its own: the difference cancels on a smooth
// state, and FP64 forms it exactly.
//
// Blocks near the limits of FP64 (subnormal values, results that under- or
// overflow) take separate conversions.  A row with an Inf or NaN in reach, or a
// diagonal entry too small for the sum's last bit beside a large value, is
// computed by h_point_fp64, one point at a time in FP64.  These choices are
// uniform over the warp.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "tdse_fixed.cuh"
#include "tdse_stencil.cuh"

namespace tdse_dev {
namespace stencil {

using namespace tdse_fx;

constexpr int kFxCols = 60;    // output columns of a strip
// A zero's exponent field is 0, and the sum's exponent T the largest of all terms',
// zeros' too: from kInLo on it is none of theirs (coefficients are below kCoupHi, an
// exponent field; the diagonal's by fx_diag_fits).
constexpr int kInLo = 256, kCoupHi = 1022 + 128;
// Diagonal entries from 2^(ec - 4) on are held exactly, and far enough above the
// sum's last bit: |D| >= 2^(ec - 4) where the encoded entry's high word reaches this.
constexpr int kDiagHigh = 1 << 25;

struct FxIn {
  const double2 *__restrict__ x;
  const long long *__restrict__ diagq;   // encoded diagonal (ok), or the FP64 diagonal's bits (!ok)
  const double *__restrict__ rj;
  const double *__restrict__ kappa;
  int N, L;
  double c1, c2, E;                      // E: the field (length gauge) or A/c (velocity gauge)
  long long c1q, c2q;                    // c1, c2 against 2^e1, 2^e2 (fx_stencil_coef)
  int e1, e2;
  int ec;                                // the diagonal's exponent
  int ok;                                // 0: the grid's coefficients do not fit, every row runs in FP64
  int k;                                 // the result is 2^k H x
  const double *__restrict__ rinv;       // velocity gauge: 1 / r_j
  double d1c;                            // velocity gauge: 1/(12 dr) (5-point) or 1/(2 dr) (3-point)
};

__device__ __forceinline__ double fx_double(uint64_t b) { return __longlong_as_double((long long)b); }

__device__ __forceinline__ double fx_diag_double(const FxIn &in, long long q) {
  if (!in.ok) return __longlong_as_double(q);
  return ldexp((double)fx_diag_value(q), in.ec + fx_diag_shift(q) - 61);
}

// 2^k (H x)(l, i) in FP64, from global memory (the rare rows; one point per call).
template <int ST, bool VG>
__device__ __noinline__ double2 h_point_fp64(const FxIn &in, int l, int i) {
  const double2 z = make_double2(0.0, 0.0);
  const size_t idx = (size_t)l * in.N + i;
  StencilIn s{};
  s.x = in.x;
  s.N = in.N;
  s.L = in.L;
  s.c1 = in.c1;
  s.c2 = in.c2;
  s.E = in.E;
  s.kappa = in.kappa;
  s.rinv = in.rinv;
  s.d1c = in.d1c;
  const double Er = VG ? 0.0 : __dmul_rn(in.E, in.rj[i]);
  const double2 prev = l > 0 ? __ldcg(in.x + idx - in.N) : z;
  const double2 next = l < in.L ? __ldcg(in.x + idx + in.N) : z;
  double2 t = h_point<ST, !VG, true>(s, in.x + (size_t)l * in.N, i, fx_diag_double(in, in.diagq[idx]), prev,
                               __ldcg(in.x + idx), next, __dmul_rn(in.kappa[l], Er), __dmul_rn(in.kappa[l + 1], Er));
  if (VG) velocity_point<ST, true>(s, l, i, prev, next, t);
  return make_double2(ldexp(t.x, in.k), ldexp(t.y, in.k));
}

// ---- staging ------------------------------------------------------------------
// A warp's rows arrive in a ring of kFxSlots slots of shared memory, each lane's
// own columns by its own cp.async copies, so a lane waits only for itself and
// no barrier is needed: of row r the operand, of the rows the warp computes
// also the diagonal and EX further vectors (the epilogue's).  While row l is
// computed row l + 2 is in flight.  Register double buffering of the operand
// alone left the epilogue's loads exposed (the top stall) and spilled.
// In the velocity gauge a slot also keeps the row's D.
constexpr int kFxSlots = 3;
template <int EX, bool VG>
constexpr int fx_slot_bytes() { return (2 + 2 * EX + 1 + (VG ? 2 : 0)) * 32 * 16; }
template <int EX, bool VG>
constexpr int fx_warp_bytes() { return kFxSlots * fx_slot_bytes<EX, VG>(); }

template <int EX>
struct FxExtra {
  const double2 *p[EX > 0 ? EX : 1];
};

// `have` false fills with zeros and reads nothing (the source is then outside the array).
__device__ __forceinline__ void cp_async16(unsigned dst, const void *src, bool have) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(have ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async8(unsigned dst, const void *src, bool have) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(have ? 8 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }

// A row of the strip in fixed point: the lane's two columns, each against its own
// largest part's exponent field (0: zero).
struct FxRow {
  int64_t X[2][2];   // [column][re, im]
  unsigned e;        // the exponent fields, column 0's in the low half
  unsigned eD;       // velocity gauge: the exponent fields of D likewise
  bool ok;           // every value of the strip finite (uniform)
};
// The half of a pair of exponent fields.
__device__ __forceinline__ int fx_half(unsigned e, int c) { return c == 0 ? (int)(e & 0xffffu) : (int)(e >> 16); }

__device__ __forceinline__ uint32_t fx_field(double v) { return (uint32_t)__double2hiint(v) & kExpMask; }
__device__ __forceinline__ int64_t fx_word(double v, uint32_t m) {
  return fx_from_words(__double2hiint(v), __double2loint(v), m);
}
__device__ __forceinline__ int64_t fx_small(double v, int e) {
  return fx_from_small(__double2hiint(v), __double2loint(v), e);
}

__device__ __forceinline__ void fx_convert(const double2 &v0, const double2 &v1, FxRow &r) {
  constexpr uint32_t kLo = (uint32_t)kExpSmall << 20;
  const uint32_t m0 = max(fx_field(v0.x), fx_field(v0.y)), m1 = max(fx_field(v1.x), fx_field(v1.y));
  r.ok = true;
  r.e = (m0 >> 20) | (m1 >> 4);
  r.eD = 0;
  if (__all_sync(0xffffffffu, min(m0, m1) >= kLo && max(m0, m1) < kExpMask)) {
    r.X[0][0] = fx_word(v0.x, m0);
    r.X[0][1] = fx_word(v0.y, m0);
    r.X[1][0] = fx_word(v1.x, m1);
    r.X[1][1] = fx_word(v1.y, m1);
  } else {
    r.ok = __all_sync(0xffffffffu, max(m0, m1) != kExpMask) != 0;
    const int e0 = max((int)(m0 >> 20), 1), e1 = max((int)(m1 >> 20), 1);
    r.X[0][0] = fx_small(v0.x, e0);
    r.X[0][1] = fx_small(v0.y, e0);
    r.X[1][0] = fx_small(v1.x, e1);
    r.X[1][1] = fx_small(v1.y, e1);
    r.e = ((r.X[0][0] | r.X[0][1]) ? e0 : 0u) | ((r.X[1][0] | r.X[1][1]) ? (unsigned)e1 << 16 : 0u);
  }
}

// V 2^(E - 1079) by the FP64 pipe's integer conversion and an addition to the exponent field.
__device__ __forceinline__ double fx_result(int64_t V, int E) {
  const double t = __ll2double_rn(V);
  const int h = __double2hiint(t);
  return __hiloint2double(h ? h + ((E - 1079) << 20) : 0, __double2loint(t));
}

// x >> n for any n >= 0
__device__ __forceinline__ int64_t fx_shr(int64_t x, int n) {
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));   // clamps the count
  return r;
}

__device__ __forceinline__ int64_t fx_shfl_up(int64_t v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ int64_t fx_shfl_down(int64_t v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// Walk rows [l0, l1) of the strip whose first output column is j0: calls
// f(idx, column, 2^k (H x), x, extra values) for every output point.  Every lane of the
// warp calls it with the same j0, l0, l1; ring: the warp's fx_warp_bytes<EX, VG>()
// of shared memory.  The operand and the extra vectors are read through L2.
template <int ST, bool VG, int EX, typename F>
__device__ __forceinline__ void walk_rows_fixed(const FxIn &in, const FxExtra<EX> &ex, unsigned char *ring, int j0,
                                                int l0, int l1, F &&f) {
  const int N = in.N, L = in.L;
  const int lane = threadIdx.x & 31;
  const int j = j0 - 2 + 2 * lane;                         // this lane's first column
  const bool have0 = j >= 0 && j < N, have1 = j + 1 >= 0 && j + 1 < N;
  const bool inner = lane >= 1 && lane <= 30;
  const bool out0 = inner && have0, out1 = inner && have1;
  // the lane's parts of a slot: 16-byte columns x0, x1, extras, diagonal pair
  unsigned char *mine = ring + lane * 16;
  const unsigned smine = (unsigned)__cvta_generic_to_shared(mine);
  constexpr int kSlot = fx_slot_bytes<EX, VG>();
  int so = (l0 - 1) * N + j;                               // the lane's element of the next row to stage
  auto stage = [&](int r, int slot) {
    const unsigned d = smine + slot * kSlot;
    if (r <= l1) {   // rows -1 and L + 1 come out as zeros
      const bool inside = r >= 0 && r <= L;
      cp_async16(d, in.x + so, have0 && inside);
      cp_async16(d + 512, in.x + so + 1, have1 && inside);
    }
    if (r >= l0 && r < l1) {
#pragma unroll
      for (int q = 0; q < EX; ++q) {
        cp_async16(d + 1024 + 1024 * q, ex.p[q] + so, out0);
        cp_async16(d + 1536 + 1024 * q, ex.p[q] + so + 1, out1);
      }
      cp_async8(d + 1024 + 1024 * EX, in.diagq + so, out0);
      cp_async8(d + 1024 + 1024 * EX + 8, in.diagq + so + 1, out1);
    }
    cp_async_commit();
    so = (int)((unsigned)so + (unsigned)N);   // past the last row it is not used
  };
  auto slot_x = [&](int slot, int c) { return *reinterpret_cast<const double2 *>(mine + slot * kSlot + 512 * c); };
  auto slow = [&](int l, int slot) {
#pragma unroll 1
    for (int c = 0; c < 2; ++c)
      if (c == 0 ? out0 : out1) {
        double2 e[EX > 0 ? EX : 1];
#pragma unroll
        for (int q = 0; q < EX; ++q)
          e[q] = *reinterpret_cast<const double2 *>(mine + slot * kSlot + 1024 + 1024 * q + 512 * c);
        f(l * N + j + c, j + c, h_point_fp64<ST, VG>(in, l, j + c), slot_x(slot, c), e);
      }
  };
  // the tables' first entries are asked for before the rows, so that their
  // latencies overlap: a warp's share is often a single row
  const double *rw = VG ? in.rinv : in.rj;
  const double rj0 = have0 ? rw[j] : 0.0, rj1 = have1 ? rw[j + 1] : 0.0;
  const double kap0 = __ldg(in.kappa + l0);
  double kap = __ldg(in.kappa + l0 + 1);                   // kappa of the next row
  stage(l0 - 1, 0);
  stage(l0, 1);
  stage(l0 + 1, 2);
  // the coupling w_j = E r_j (velocity gauge: E / r_j) of the lane's columns
  const double w0 = __dmul_rn(in.E, rj0), w1 = __dmul_rn(in.E, rj1);
  const double wd = VG ? __dmul_rn(in.E, in.d1c) : 0.0;    // velocity gauge: the derivative's coefficient
  const bool all_ok =
      in.ok && __all_sync(0xffffffffu, max(max(fx_field(w0), fx_field(w1)), fx_field(wd)) < (uint32_t)kCoupHi << 20) != 0;
  const int we0 = max((int)(fx_field(w0) >> 20), 1), we1 = max((int)(fx_field(w1) >> 20), 1);
  const int ew[2] = {we0 - 1022, we1 - 1022};              // w = W 2^(ew - 60)
  const Limb W[2] = {fx_limbs(fx_small(w0, we0)), fx_limbs(fx_small(w1, we1))};
  // length gauge: a = kappa_l w = A 2^(ew - 61); velocity gauge: a = kappa_l l w =
  // A 2^(ew + el - 61) with 2^el > l, and d = kappa_l E d1c = D 2^(ed - 61)
  const int wde = max((int)(fx_field(wd) >> 20), 1), ed = wde - 1022;
  const Limb WD = fx_limbs(VG ? fx_small(wd, wde) : 0);
  auto coupling = [&](int l, double kappa, Limb (&a)[2], Limb &d, int &el) {
    const int64_t K = fx_coef((uint64_t)__double_as_longlong(kappa), 0);
    Limb kp = fx_limbs(K);
    if (VG) {
      d = fx_limbs(fx_coef_product(kp, WD));
      el = 32 - __clz(l | 1);
      // K l / 2^el, odd: no limb is -2^31, so that the next row can negate it
      kp = fx_limbs((int64_t)(__umul64hi((uint64_t)K << 2, (uint64_t)l << (64 - el)) >> 2));
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) a[c] = fx_limbs(fx_coef_product(kp, W[c]) | (VG ? 1 : 0));
  };
  // velocity gauge: the differences D of a row into the slot, each column's against
  // the largest exponent of its terms and then brought to 58 bits, so that what
  // cancels costs no bits: D = 8 Q (5-point) or Q (3-point)
  auto differences = [&](FxRow &r, int slot) {
    const unsigned u = __shfl_up_sync(0xffffffffu, r.e, 1), d = __shfl_down_sync(0xffffffffu, r.e, 1);
    const int eA = fx_half(r.e, 0), eB = fx_half(r.e, 1), eU = fx_half(u, 1), eV = fx_half(d, 0);
    const int eUA = fx_half(u, 0), eVB = fx_half(d, 1);
    int b0 = max(eU, eB), b1 = max(eA, eV);
    if (ST == 5) {
      b0 = max(b0, max(eUA, eV));
      b1 = max(b1, max(eU, eVB));
    }
    int64_t Q[2][2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int64_t A = r.X[0][p], B = r.X[1][p], lB = fx_shfl_up(B), rA = fx_shfl_down(A);
      Q[0][p] = fx_shr(B, b0 - eB) - fx_shr(lB, b0 - eU);
      Q[1][p] = fx_shr(rA, b1 - eV) - fx_shr(A, b1 - eA);
      if (ST == 5) {
        const int64_t lA = fx_shfl_up(A), rB = fx_shfl_down(B);
        Q[0][p] -= (fx_shr(rA, b0 - eV) - fx_shr(lA, b0 - eUA)) >> 3;
        Q[1][p] -= (fx_shr(rB, b1 - eVB) - fx_shr(lB, b1 - eU)) >> 3;
      }
    }
    constexpr int k8 = ST == 5 ? 3 : 0;
    const int n0 = min(fx_lead(Q[0][0], Q[0][1]), b0 + k8 - 1), n1 = min(fx_lead(Q[1][0], Q[1][1]), b1 + k8 - 1);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const longlong2 D = make_longlong2(fx_bring(Q[0][p], n0), fx_bring(Q[1][p], n1));
      *reinterpret_cast<longlong2 *>(mine + slot * kSlot + kSlot - 1024 + 512 * p) = D;
    }
    r.eD = ((Q[0][0] | Q[0][1]) ? (unsigned)(b0 - n0 + k8) : 0u) |
           ((Q[1][0] | Q[1][1]) ? (unsigned)(b1 - n1 + k8) << 16 : 0u);
  };
  const Limb k1 = fx_limbs(in.c1q), k2 = fx_limbs(in.c2q);
  Limb acur[2], anext[2], dcur = {0, 0}, dnext = {0, 0};
  int lcur = 0, lnext = 0;
  coupling(l0, kap0, acur, dcur, lcur);
  if (VG)
#pragma unroll
    for (int c = 0; c < 2; ++c) acur[c] = Limb{-acur[c].h, -acur[c].l};
  FxRow prev, cur, next;
  cp_async_wait<1>();
  fx_convert(slot_x(0, 0), slot_x(0, 1), prev);
  fx_convert(slot_x(1, 0), slot_x(1, 1), cur);
  if (VG) {
    differences(prev, 0);
    differences(cur, 1);
  }
  stage(l0 + 2, 0);
  // T between these: nothing near FP64's limits
  const int tlo = max(kInLo, kOutLo - in.k), thi = kOutHi - in.k;
  int s0 = 1, s1 = 2;                                      // slots of rows l and l + 1
#pragma unroll 1
  for (int l = l0; l < l1; ++l) {
    cp_async_wait<1>();
    fx_convert(slot_x(s1, 0), slot_x(s1, 1), next);
    if (VG) differences(next, s1);
    coupling(l + 1, kap, anext, dnext, lnext);
    if (l + 1 < l1) kap = __ldg(in.kappa + l + 2);
    const unsigned char *body = mine + s0 * kSlot;
    const longlong2 dq = *reinterpret_cast<const longlong2 *>(body + 1024 + 1024 * EX);
    const unsigned u = __shfl_up_sync(0xffffffffu, cur.e, 1), d = __shfl_down_sync(0xffffffffu, cur.e, 1);
    // columns: UA UB | A B | VA VB
    const int eUA = fx_half(u, 0), eUB = fx_half(u, 1), eA = fx_half(cur.e, 0), eB = fx_half(cur.e, 1);
    const int eVA = fx_half(d, 0), eVB = fx_half(d, 1);
    const int near[2] = {max(eUB, eB), max(eA, eVA)};
    const int far[2] = {ST == 5 ? max(eUA, eVA) : 0, ST == 5 ? max(eUB, eVB) : 0};
    // T: exponent of a point's sum, the largest of its own terms'
    int T[2], td[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      td[c] = in.ec + fx_diag_shift(c == 0 ? dq.x : dq.y);
      T[c] = max(near[c] + in.e1, (c == 0 ? eA : eB) + td[c]);
      if (ST == 5) T[c] = max(T[c], far[c] + in.e2);
      T[c] = max(T[c], max(fx_half(prev.e, c) + lcur, fx_half(next.e, c) + lnext) + ew[c]);
      if (VG) T[c] = max(T[c], max(fx_half(prev.eD, c), fx_half(next.eD, c)) + ed);
    }
    bool fixed = all_ok && prev.ok && cur.ok && next.ok, limits = false, zero = false;   // uniform
    const int h0 = (int)(dq.x >> 32), h1 = (int)(dq.y >> 32);
    if (fixed && !__all_sync(0xffffffffu, !inner || (min(T[0], T[1]) >= tlo && max(T[0], T[1]) <= thi &&
                                                     min(abs(h0), abs(h1)) >= kDiagHigh))) {
      // near FP64's limits, zeros, small diagonal entries: T again, of the terms that are not zero
      auto term = [](int e, int c) { return e ? e + c : kNone; };
      bool good = true, range = true;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int e = c == 0 ? eA : eB;
        T[c] = max(term(near[c], in.e1), term(e, td[c]));
        if (ST == 5) T[c] = max(T[c], term(far[c], in.e2));
        T[c] = max(T[c], max(term(fx_half(prev.e, c), lcur + ew[c]), term(fx_half(next.e, c), lnext + ew[c])));
        if (VG) T[c] = max(T[c], max(term(fx_half(prev.eD, c), ed), term(fx_half(next.eD, c), ed)));
        if (c == 0 ? out0 : out1) {
          good = good && (abs(c == 0 ? h0 : h1) >= kDiagHigh || e <= near[c]);
          range = range && (T[c] == kNone || (T[c] >= kOutLo - in.k && T[c] <= thi));
        }
      }
      fixed = __all_sync(0xffffffffu, good) != 0;
      limits = !__all_sync(0xffffffffu, range);
      zero = __all_sync(0xffffffffu, (prev.e | cur.e | next.e) == 0) != 0;   // a tail that has underflowed, an empty wave
    }
    if (fixed) {
      const unsigned char *pd = mine + (kFxSlots - s0 - s1) * kSlot + kSlot - 1024, *nd = mine + s1 * kSlot + kSlot - 1024;
      const Limb kd[2] = {fx_limbs(fx_diag_value(dq.x)), fx_limbs(fx_diag_value(dq.y))};
      double t[2][2] = {};
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        if (zero) break;
        const int64_t A = cur.X[0][p], B = cur.X[1][p], UB = fx_shfl_up(B), VA = fx_shfl_down(A);
        int64_t UA = 0, VB = 0;
        if (ST == 5) {
          UA = fx_shfl_up(A);
          VB = fx_shfl_down(B);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {   // every operand is moved to T before its product
          int64_t hh = 0, mm = kHalf >> kFineBits;
          const int t1 = T[c] - in.e1, t2 = T[c] - in.e2;
          fx_mac(fx_limbs(c == 0 ? fx_shr(UB, t1 - eUB) + fx_shr(B, t1 - eB) : fx_shr(A, t1 - eA) + fx_shr(VA, t1 - eVA)),
                 k1, hh, mm);
          if (ST == 5)
            fx_mac(fx_limbs(c == 0 ? fx_shr(UA, t2 - eUA) + fx_shr(VA, t2 - eVA)
                                   : fx_shr(UB, t2 - eUB) + fx_shr(VB, t2 - eVB)), k2, hh, mm);
          fx_mac(fx_limbs(fx_shr(c == 0 ? A : B, T[c] - td[c] - (c == 0 ? eA : eB))), kd[c], hh, mm);
          const int sp = T[c] - ew[c] - lcur - fx_half(prev.e, c), sn = T[c] - ew[c] - lnext - fx_half(next.e, c);
          if (!VG) {
            fx_mac(fx_limbs(fx_shr(prev.X[c][p], sp)), acur[c], hh, mm);
            fx_mac(fx_limbs(fx_shr(next.X[c][p], sn)), anext[c], hh, mm);
          } else {   // -i (A/c) w: the real part takes +w's imaginary part, the imaginary part -w's real part
            int64_t ch = 0, cm = 0;
            const int64_t *dp = reinterpret_cast<const int64_t *>(pd + 512 * (1 - p)) + c;
            const int64_t *dn = reinterpret_cast<const int64_t *>(nd + 512 * (1 - p)) + c;
            fx_mac(fx_limbs(fx_shr(prev.X[c][1 - p], sp)), acur[c], ch, cm);
            fx_mac(fx_limbs(fx_shr(next.X[c][1 - p], sn)), anext[c], ch, cm);
            fx_mac(fx_limbs(fx_shr(*dp, T[c] - ed - fx_half(prev.eD, c))), dcur, ch, cm);
            fx_mac(fx_limbs(fx_shr(*dn, T[c] - ed - fx_half(next.eD, c))), dnext, ch, cm);
            hh = p == 0 ? hh + ch : hh - ch;
            mm = p == 0 ? mm + cm : mm - cm;
          }
          const int64_t V = fx_value(hh, mm, kFineBits);
          const int E = T[c] + in.k - kFineBits;
          t[c][p] = limits ? ldexp(fx_double(fx_to_bits(V, 1000)), V ? E - 1000 : 0) : fx_result(V, E);
        }
      }
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (c == 0 ? out0 : out1) {
          double2 e[EX > 0 ? EX : 1];
#pragma unroll
          for (int q = 0; q < EX; ++q) e[q] = *reinterpret_cast<const double2 *>(body + 1024 + 1024 * q + 512 * c);
          f(l * N + j + c, j + c, make_double2(t[c][0], t[c][1]), *reinterpret_cast<const double2 *>(body + 512 * c),
            e);
        }
    } else {
      slow(l, s0);
    }
    stage(l + 3, s0);
    const int s2 = kFxSlots - s0 - s1;
    s0 = s1;
    s1 = s2;
    prev = cur;
    cur = next;
#pragma unroll
    for (int c = 0; c < 2; ++c) acur[c] = VG ? Limb{-anext[c].h, -anext[c].l} : anext[c];
    dcur = dnext;
    lcur = lnext;
  }
  cp_async_wait<0>();   // the ring is free for the next call
}

// Visit this warp's share of the strips' row segments (strip-major): f(j0, l0,
// l1), by every lane.  Warp k of block b of a grid of B blocks has number
// k B + b: the first of the numbers take one segment more, and so do as many
// warps of every block.
template <typename F>
__device__ __forceinline__ void for_my_strips(const FxIn &in, F &&f) {
  const unsigned Lp1 = (unsigned)in.L + 1u, T = (((unsigned)in.N + kFxCols - 1u) / kFxCols) * Lp1;
  const unsigned W = gridDim.x * (blockDim.x >> 5), w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const unsigned q = T / W, r = T - q * W;
  unsigned s = w * q + min(w, r);
  const unsigned s_end = s + q + (w < r ? 1u : 0u);
  while (s < s_end) {
    const unsigned sg = s / Lp1, l0 = s - sg * Lp1, l1 = min(Lp1, l0 + (s_end - s));
    f((int)(sg * kFxCols), (int)l0, (int)l1);
    s += l1 - l0;
  }
}

}  // namespace stencil
}  // namespace tdse_dev
