// FP64 kernels of the finite-difference TDSE path (sm_103a).
//
// Every stencil kernel evaluates the Hamiltonian of Eq. (h_matrix), in the length gauge
// (arXiv 1308.1856, Sec. 2):
//   (H x)_{l,j} = D_{l,j} x_{l,j} + c1 (x_{l,j-1} + x_{l,j+1}) [+ c2 (x_{l,j-2} + x_{l,j+2})]
//               + E r_j (kappa_l x_{l-1,j} + kappa_{l+1} x_{l+1,j})
// with D_{l,j} = c0 + l(l+1)/(2 r_j^2) + V(r_j) read from a table, H real and
// symmetric, so the real and imaginary parts go through the same real operator.
//
// The operator runs in the fixed-point walker (tdse_walk_fixed.cuh).  An FP64
// instruction of a warp takes its SM sub-partition 64 cycles, so the 15 of a
// point's H x (velocity gauge: 34) bounded these kernels; in fixed point the
// operator runs on the integer pipe and only the epilogue is FP64.  The (L+1)
// rows of the strips of kFxCols columns form one strip-major sequence of row
// segments; warp w of the persistent grid takes a contiguous, balanced range of
// it (for_my_strips).  The warps' numbers run across the blocks, so that the
// warps with one segment more are spread evenly over the SMs.
//
// All in FP64 run the Taylor and RK4 stages of length-gauge grids that fit the
// one-launch cluster path, whose states are bitwise these, and every kernel of a
// grid without the fixed-point form (coefficients that do not fit, or no memory
// for its diagonal; OperatorView::plain): in segments of 32 radial
// points of one partial wave, ordered radial-group-major, a contiguous balanced
// range for each warp (warp_range).  A lane owns one radial index j and walks l
// upwards keeping x_{l-1,j}, x_{l,j}, x_{l+1,j} in registers; the arithmetic is
// written with explicit __dmul_rn / __dadd_rn / __fma_rn.
// H x of 512,000 points on a grid whose potential does not fit: 19 us in these
// registers, velocity gauge 45 us; point by point from L2 in the fixed-point walker 35
// and 62 us.
#include <cuda_runtime.h>

#include <type_traits>

#include "tdse_device_common.cuh"
#include "tdse_stencil.cuh"
#include "tdse_walk_fixed.cuh"
#include "tdse_combine_fixed.cuh"
#include "tdse_internal.cuh"

namespace tdse_dev {

namespace {

using namespace common;
using namespace stencil;

// Visit this warp's share of the 32-point row segments (see the file header).
template <int ST, bool VG, typename F>
__device__ __forceinline__ void for_my_segments(const StencilIn &in, F &&f) {
  const int lane = threadIdx.x & 31;
  const int Lp1 = in.L + 1;
  const long long NJ = (in.N + 31) >> 5;
  long long s, s_end;
  warp_range(NJ * Lp1, s, s_end);
  while (s < s_end) {
    const int jg = (int)((unsigned)s / (unsigned)Lp1);
    const int l0 = (int)(s - (long long)jg * Lp1);
    const long long left = s_end - s;
    const int l1 = (left < (long long)(Lp1 - l0)) ? l0 + (int)left : Lp1;
    const int i = jg * 32 + lane;
    if (i < in.N) walk_rows<ST, VG>(in, i, l0, l1, f);
    s += l1 - l0;
  }
}

// How a stencil kernel walks the grid: in fixed point or in FP64, in the length or
// the velocity gauge.
enum Walk { kFixed, kFixedVG, kPlain, kPlainVG };
constexpr bool is_plain(int walk) { return walk == kPlain || walk == kPlainVG; }
template <int WALK>
using OpIn = std::conditional_t<is_plain(WALK), StencilIn, FxIn>;
// Blocks an SM: one of 16 warps with 128 registers a thread and its rings in
// fixed point, two of 64 registers in FP64.
template <int WALK>
constexpr int kOpBlocksPerSM = is_plain(WALK) ? kStencilBlocksPerSM : 1;

// Call f(idx, i, H x, x, extra values) at every point this thread owns.
template <int ST, int WALK, int EX, typename F>
__device__ __forceinline__ void for_my_points(const OpIn<WALK> &in, const FxExtra<EX> &ex, F &&f) {
  if constexpr (is_plain(WALK)) {
    for_my_segments<ST, WALK == kPlainVG>(in, [&](int i, size_t idx, double2 t, double2 u) {
      double2 e[EX > 0 ? EX : 1];
#pragma unroll
      for (int q = 0; q < EX; ++q) e[q] = ex.p[q][idx];
      f((int)idx, i, t, u, e);
    });
  } else {
    extern __shared__ __align__(16) unsigned char fx_smem[];
    unsigned char *ring = fx_smem + (threadIdx.x >> 5) * fx_warp_bytes<EX, WALK == kFixedVG>();
    for_my_strips(in, [&](int j0, int l0, int l1) {
      walk_rows_fixed<ST, WALK == kFixedVG, EX>(in, ex, ring, j0, l0, l1, f);
    });
  }
}

// ---------------------------------------------------------------------------
// y = H(E) x
template <int ST, int WALK>
__global__ void __launch_bounds__(kBlockJ, kOpBlocksPerSM<WALK>)
    apply_h_kernel(OpIn<WALK> in, double2 *__restrict__ y) {
  for_my_points<ST, WALK, 0>(in, FxExtra<0>{}, [&](int idx, int, double2 t, double2, const double2 (&)[1]) {
    y[idx] = t;
  });
}

// Horner stage of the Taylor polynomial (Eq. (Taylor)):
//   v_out = psi + (-i s) H v_in,  s = dt / k   (IMAG: psi - s H v_in, Sec. 3's
//   imaginary-time propagation).
// The last stage (k = 1, FIN) writes psi itself and applies the absorber
// mask; the other stages carry no mask code at all (a predicated-off FP64
// instruction still takes its issue slot on the FP64 pipe).
template <int ST, bool IMAG, int WALK, bool FIN>
__global__ void __launch_bounds__(kBlockJ, kOpBlocksPerSM<WALK>)
    taylor_stage_kernel(OpIn<WALK> in, double s, const double2 *psi, double2 *out, const double *__restrict__ mask,
                        int mask_start) {
  pdl_wait();
  FxExtra<1> ex;
  ex.p[0] = psi;
  for_my_points<ST, WALK, 1>(in, ex, [&](int idx, int i, double2 t, double2, const double2 (&e)[1]) {
    const bool masked = FIN && i >= mask_start;
    double2 o;
    if (IMAG) {
      o.x = __fma_rn(-s, t.x, e[0].x);
      o.y = __fma_rn(-s, t.y, e[0].y);
    } else {
      o.x = __fma_rn(s, t.y, e[0].x);     // (-i s)(tx + i ty) = s ty - i s tx
      o.y = __fma_rn(-s, t.x, e[0].y);
    }
    if (masked) { const double mv = mask[i]; o.x = __dmul_rn(mv, o.x); o.y = __dmul_rn(mv, o.y); }
    out[idx] = o;
  });
  pdl_trigger();
}

// A stage of classic RK4 (Eq. (RKDeriv)) with k = -i H(t_n + c dt) g:
//   PART 0, stage 1 (g = psi):  g_next = psi + ca k,  acc = psi + cb k
//   PART 1, stages 2 and 3:     g_next = psi + ca k,  acc = acc + cb k
//   PART 2, stage 4:            psi    = acc + cb k, then the absorber mask.
// IMAG: k = -H g (imaginary time) instead of -i H g.
template <int ST, bool IMAG, int WALK, int PART>
__global__ void __launch_bounds__(kBlockJ, kOpBlocksPerSM<WALK>)
    rk_stage_kernel(OpIn<WALK> in, double ca, double cb, const double2 *psi, double2 *acc, double2 *g_next,
                    double2 *psi_out, const double *__restrict__ mask, int mask_start) {
  pdl_wait();
  constexpr int EX = PART == 0 ? 0 : (PART == 1 ? 2 : 1);
  FxExtra<EX> ex;
  if (PART > 0) ex.p[0] = acc;
  if constexpr (PART == 1) ex.p[1] = psi;
  for_my_points<ST, WALK, EX>(in, ex, [&](int idx, int i, double2 t, double2 u, const double2 (&e)[EX > 0 ? EX : 1]) {
    // c k with k = -i t:  (c t.y, -c t.x);  with k = -t:  (-c t.x, -c t.y)
    auto add = [&](double c, double2 base) {
      return IMAG ? make_double2(__fma_rn(-c, t.x, base.x), __fma_rn(-c, t.y, base.y))
                  : make_double2(__fma_rn(c, t.y, base.x), __fma_rn(-c, t.x, base.y));
    };
    if constexpr (PART == 0) {
      g_next[idx] = add(ca, u);
      acc[idx] = add(cb, u);
    } else if constexpr (PART == 1) {
      g_next[idx] = add(ca, e[1]);
      acc[idx] = add(cb, e[0]);
    } else {
      double2 o = add(cb, e[0]);
      if (i >= mask_start) { const double mv = mask[i]; o.x = __dmul_rn(mv, o.x); o.y = __dmul_rn(mv, o.y); }
      psi_out[idx] = o;
    }
  });
  pdl_trigger();
}

// Stage a.stage of a general explicit Runge-Kutta method (appendix
// "Runge-Kutta"); see RkStageArgs.  NK = a.stage + 1 terms and MODE are
// compile-time, so no FP64 instruction is issued for absent terms (a
// predicated-off FP64 instruction still takes its FP64 issue slot):
//   MODE 0: an inner stage (k_i and g_{i+1} out);
//   MODE 1: the last stage (psi, Delta and the sigma partial);
//   MODE 2: the last stage of a first-same-as-last tableau (b_{s-1} = 0 and
//           a_{s-1,j} = b_j): psi_new is the stage's own input g_{s-1}, which
//           the previous stage summed in the same order with the same
//           coefficients, so only Delta is formed.
// The slopes of the earlier stages are read pointwise and combined in stage
// order, the new slope k_i = -i H g_i last, so the sums round in the same
// order as the oracle's.  psi (or, in MODE 2, k_0) and the first slope come
// through the walker's ring, which has room for two vectors; further slopes are
// loaded where they are used.
template <int ST, int WALK, int NK, int MODE>
__global__ void __launch_bounds__(kBlockJ, kOpBlocksPerSM<WALK>)
    rk_general_stage_kernel(OpIn<WALK> in, RkStageArgs a, const double2 *psi, const double *__restrict__ mask,
                            int mask_start, Reduction *red, double S) {
  constexpr bool LAST = MODE != 0;
  constexpr bool FSAL = MODE == 2;
  constexpr int VECS = FSAL ? NK - 1 : NK;          // psi unless FSAL, then the earlier slopes
  constexpr int EX = VECS < 2 ? VECS : 2;
  constexpr int KOFF = FSAL ? 0 : 1;                // slope j is vector j + KOFF
  __shared__ double sh[kBlockJ / 32 + 1];
  double acc = 0.0;
  pdl_wait();
  FxExtra<EX> ex;
#pragma unroll
  for (int q = 0; q < EX; ++q) ex.p[q] = (q < KOFF) ? psi : a.k[q - KOFF];
  for_my_points<ST, WALK, EX>(in, ex, [&](int idx, int r, double2 t, double2 u, const double2 (&e)[EX > 0 ? EX : 1]) {
    const double2 ki = make_double2(t.y, -t.x);   // -i (tx + i ty)
    double2 kj[NK > 1 ? NK - 1 : 1];
#pragma unroll
    for (int j = 0; j < NK - 1; ++j) kj[j] = (j + KOFF < EX) ? e[j + KOFF] : a.k[j][idx];
    double2 o = FSAL ? u : e[0];
    double2 d = make_double2(0.0, 0.0);
#pragma unroll
    for (int j = 0; j < NK - 1; ++j) {
      if (!FSAL) {
        o.x = __fma_rn(a.coef[j], kj[j].x, o.x);
        o.y = __fma_rn(a.coef[j], kj[j].y, o.y);
      }
      if (LAST) {
        d.x = __fma_rn(a.dcoef[j], kj[j].x, d.x);
        d.y = __fma_rn(a.dcoef[j], kj[j].y, d.y);
      }
    }
    if (!FSAL) {
      o.x = __fma_rn(a.coef[NK - 1], ki.x, o.x);
      o.y = __fma_rn(a.coef[NK - 1], ki.y, o.y);
    }
    if (!LAST) {
      a.k_out[idx] = ki;
      a.g_out[idx] = o;
    } else {
      d.x = __fma_rn(a.dcoef[NK - 1], ki.x, d.x);
      d.y = __fma_rn(a.dcoef[NK - 1], ki.y, d.y);
      acc = __fma_rn(d.x, d.x, acc);
      acc = __fma_rn(d.y, d.y, acc);
      if (r >= mask_start) { const double mv = mask[r]; o.x = __dmul_rn(mv, o.x); o.y = __dmul_rn(mv, o.y); }
      a.psi_out[idx] = o;
    }
  });
  pdl_trigger();
  if (LAST && publish_block_partial(acc, red, sh)) {
    const double s = reduce_partials(red, gridDim.x, sh);
    if (threadIdx.x == 0) {
      *a.sigma += sqrt(s / S);
      if (!isfinite(s)) atomicOr(a.status, kStatusNonFinite);
    }
  }
}

// Lanczos iteration j, first half (Appendix "Lanczos methods"):
//   z = s_j H U_j - ratio_j U_{j-1},  alpha_j from sum Re(U_j^* z)
// with s_j the power of two at or below sigma_j (step_scale; the grid
// reduction's last block stores the scalars).  EX = 1 where U_{j-1} exists.
template <int ST, int WALK, int EX>
__global__ void __launch_bounds__(kBlockJ, kOpBlocksPerSM<WALK>)
    lanczos_a_kernel(OpIn<WALK> in, int j, const double2 *__restrict__ uprev, double2 *__restrict__ z, Reduction *red,
                     LanczosScalars *ls) {
  __shared__ double sh[kBlockJ / 32 + 1];
  pdl_wait();
  const StepScale sc = step_scale(ls->sigma[j]);
  const double cprev = EX > 0 ? ls->ratio[j] : 0.0;
  double acc = 0.0;
  FxExtra<EX> ex;
  if (EX > 0) ex.p[0] = uprev;
  if constexpr (!is_plain(WALK)) in.k = sc.k;
  for_my_points<ST, WALK, EX>(in, ex, [&](int idx, int, double2 t, double2 u, const double2 (&e)[1]) {
    if (is_plain(WALK)) t = make_double2(__dmul_rn(sc.s, t.x), __dmul_rn(sc.s, t.y));
    double2 o = t;
    if (EX > 0) {
      o.x = __fma_rn(-cprev, e[0].x, t.x);
      o.y = __fma_rn(-cprev, e[0].y, t.y);
    }
    z[idx] = o;
    acc = __fma_rn(u.x, o.x, acc);
    acc = __fma_rn(u.y, o.y, acc);
  });
  pdl_trigger();
  if (publish_block_partial(acc, red, sh)) {
    const double s = reduce_partials(red, gridDim.x, sh);
    if (threadIdx.x == 0) store_alpha(ls, j, s);
  }
}

// Elementwise kernels: persistent grid; each warp takes a contiguous, balanced
// range of the groups of 32 consecutive elements (warp_range).

template <typename F>
__device__ __forceinline__ void for_my_groups(size_t G, F &&f) {
  const int lane = threadIdx.x & 31;
  long long g0, g1;
  warp_range((long long)((G + 31) >> 5), g0, g1);
  for (long long gi = g0; gi < g1; ++gi) {
    const size_t idx = (size_t)gi * 32 + lane;
    if (idx < G) f(idx);
  }
}

// Up to kUnroll groups of this warp's range are loaded before any of them is
// used, so their memory latencies overlap.
constexpr int kUnroll = 4;

// Lanczos iteration j, second half: U_{j+1} = z - alpha_j s_j U_j and its norm (beta_j).
__global__ void __launch_bounds__(kElemThreads, kElemBlocksPerSM)
    lanczos_b_kernel(size_t G, int j, const double2 *__restrict__ z, const double2 *__restrict__ u,
                     double2 *__restrict__ unext, Reduction *red, LanczosScalars *ls) {
  __shared__ double sh[kElemThreads / 32 + 1];
  pdl_wait();
  const double c = ls->acoef[j];
  double acc0 = 0.0, acc1 = 0.0;
  const int lane = threadIdx.x & 31;
  long long g0, g1;
  warp_range((long long)((G + 31) >> 5), g0, g1);
  for (long long gb = g0; gb < g1; gb += kUnroll) {
    double2 zz[kUnroll], uu[kUnroll];
#pragma unroll
    for (int r = 0; r < kUnroll; ++r) {
      const size_t idx = (size_t)(gb + r) * 32 + lane;
      const bool ok = (gb + r < g1) && idx < G;
      zz[r] = ok ? z[idx] : make_double2(0.0, 0.0);
      uu[r] = ok ? u[idx] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int r = 0; r < kUnroll; ++r) {
      const size_t idx = (size_t)(gb + r) * 32 + lane;
      if ((gb + r < g1) && idx < G) {
        const double2 o = make_double2(__fma_rn(c, uu[r].x, zz[r].x), __fma_rn(c, uu[r].y, zz[r].y));
        unext[idx] = o;
        acc0 = __fma_rn(o.x, o.x, acc0);
        acc1 = __fma_rn(o.y, o.y, acc1);
      }
    }
  }
  pdl_trigger();
  if (publish_block_partial(acc0 + acc1, red, sh)) {
    const double s = reduce_partials(red, gridDim.x, sh);
    if (threadIdx.x == 0) store_beta(ls, j, s);
  }
}

// ||x||^2 -> Lanczos start scalars (sigma_0 = 1/||psi||, psinorm) and the
// non-finite status bit.
__global__ void __launch_bounds__(kElemThreads, kElemBlocksPerSM)
    norm_kernel(size_t G, const double2 *__restrict__ x, Reduction *red, LanczosScalars *ls,
                int *status) {
  __shared__ double sh[kElemThreads / 32 + 1];
  pdl_wait();
  double acc0 = 0.0, acc1 = 0.0;
  const int lane = threadIdx.x & 31;
  long long g0, g1;
  warp_range((long long)((G + 31) >> 5), g0, g1);
  for (long long gb = g0; gb < g1; gb += kUnroll) {
    double2 v[kUnroll];
#pragma unroll
    for (int r = 0; r < kUnroll; ++r) {
      const size_t idx = (size_t)(gb + r) * 32 + lane;
      v[r] = ((gb + r < g1) && idx < G) ? x[idx] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int r = 0; r < kUnroll; ++r) {
      acc0 = __fma_rn(v[r].x, v[r].x, acc0);
      acc1 = __fma_rn(v[r].y, v[r].y, acc1);
    }
  }
  pdl_trigger();
  if (publish_block_partial(acc0 + acc1, red, sh)) {
    const double s = reduce_partials(red, gridDim.x, sh);
    if (threadIdx.x == 0) {
      red->normsq = s;
      norm_and_inverse(s, ls->psinorm, ls->sigma[0]);
      if (!isfinite(s)) atomicOr(status, kStatusNonFinite);
    }
  }
}

// Imaginary time (Sec. 3): the squared norm before a step, then after it the
// energy estimate and the renormalisation of psi.
__global__ void imag_begin_kernel(const Reduction *red, double dr, double *imag) {
  imag[0] = dr * red->normsq;
}

__global__ void __launch_bounds__(kElemThreads, kElemBlocksPerSM)
    imag_normalize_kernel(size_t G, double2 *psi, const Reduction *red, double dr, double dt,
                          double *imag) {
  const double n2 = dr * red->normsq;
  const double sc = (n2 > 0.0) ? 1.0 / sqrt(n2) : 0.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) imag[1] = -log(n2 / imag[0]) / (2.0 * dt);
  for_my_groups(G, [&](size_t idx) {
    const double2 v = psi[idx];
    psi[idx] = make_double2(__dmul_rn(sc, v.x), __dmul_rn(sc, v.y));
  });
}

// psi_new = sum_{j<k} coef_j U_j  (U_0 = psi, read and written in place by
// the same thread), then the absorber mask and ||psi_new||^2 for the next step.
// The sum in fixed point (tdse_combine_fixed.cuh), 128 registers a thread for
// its loads in flight.
__global__ void __launch_bounds__(kElemThreads, 1)
    lanczos_combine_kernel(size_t G, int N, double2 *psi, const double2 *__restrict__ work,
                           size_t stride, const double *__restrict__ mask, int mask_start,
                           Reduction *red, LanczosScalars *ls, int *status) {
  __shared__ double sh[kElemThreads / 32 + 1];
  __shared__ CbTable tab;
  pdl_wait();
  if (threadIdx.x < 32) cb_setup(tab, ls);
  __syncthreads();
  double acc = 0.0;
  const int lane = threadIdx.x & 31;
  long long g0, g1;
  warp_range((long long)((G + 31) >> 5), g0, g1);
  for (long long gi = g0; gi < g1; ++gi) {
    const size_t idx = (size_t)gi * 32 + lane;
    const bool ok = idx < G;
    double2 o = cb_sum(tab, [&](int j) {
      return ok ? (j == 0 ? psi[idx] : work[(size_t)(j - 1) * stride + idx]) : make_double2(0.0, 0.0);
    });
    if (!ok) continue;
    const int jr = (int)((unsigned)idx % (unsigned)N);
    if (jr >= mask_start) {
      const double mv = mask[jr];
      o.x = __dmul_rn(mv, o.x);
      o.y = __dmul_rn(mv, o.y);
    }
    psi[idx] = o;
    acc = __fma_rn(o.x, o.x, acc);
    acc = __fma_rn(o.y, o.y, acc);
  }
  pdl_trigger();
  if (publish_block_partial(acc, red, sh)) {
    const double s = reduce_partials(red, gridDim.x, sh);
    if (threadIdx.x == 0) {
      red->normsq = s;
      norm_and_inverse(s, ls->psinorm, ls->sigma[0]);
      if (!isfinite(s)) atomicOr(status, kStatusNonFinite);
    }
  }
}

// The diagonal in the fixed-point walker's encoding.
__global__ void __launch_bounds__(256) fx_diag_kernel(const double *__restrict__ diag, size_t G, int ec,
                                                      long long *__restrict__ diagq) {
  for (size_t q = (size_t)blockIdx.x * 256 + threadIdx.x; q < G; q += (size_t)gridDim.x * 256)
    diagq[q] = fx_encode_diag((uint64_t)__double_as_longlong(diag[q]), ec);
}

// Observables (Sec. 4): per block of row l, partial sums of
//   q0: sum |f|^2, q1: sum_{r_j <= r_b} |f|^2, q2: sum r_j Re(conj(f_l) f_{l+1}),
//   q3, q4: sum conj(ref_j) f_{0,j} (row 0 only).
// Partials are laid out [q][row][bx]; the last block combines them in index
// order into out = {norm, dipole, yield, p_ground, l_pop[0..L]}.
constexpr int kObsThreads = 256;
constexpr int kObsQ = 5;

__global__ void __launch_bounds__(kObsThreads)
    observables_kernel(const double2 *__restrict__ psi, const double2 *__restrict__ ref0,
                       const double *__restrict__ rj, const double *__restrict__ kappa,
                       int N, int L, double dr, double r_b, double *partials,
                       unsigned *ticket, double *out) {
  __shared__ double sh[kObsThreads / 32 + 1];
  __shared__ unsigned s_last;
  const int l = blockIdx.y;
  const int nbx = gridDim.x;
  double q[kObsQ] = {0.0, 0.0, 0.0, 0.0, 0.0};
  for (int i = blockIdx.x * kObsThreads + threadIdx.x; i < N; i += nbx * kObsThreads) {
    const size_t idx = (size_t)l * N + i;
    const double2 f = psi[idx];
    const double a = __fma_rn(f.x, f.x, __dmul_rn(f.y, f.y));
    const double r = rj[i];
    q[0] += a;
    if (r <= r_b) q[1] += a;
    if (l < L) {
      const double2 g = psi[idx + N];
      q[2] = __fma_rn(r, __fma_rn(f.x, g.x, __dmul_rn(f.y, g.y)), q[2]);
    }
    if (l == 0 && ref0) {
      const double2 c = ref0[i];
      q[3] += __fma_rn(c.x, f.x, __dmul_rn(c.y, f.y));    // Re(conj(c) f)
      q[4] += __fma_rn(c.x, f.y, __dmul_rn(-c.y, f.x));   // Im(conj(c) f)
    }
  }
  const size_t nb = (size_t)nbx * (L + 1);
  const size_t bid = (size_t)l * nbx + blockIdx.x;
  for (int k = 0; k < kObsQ; ++k) {
    const double b = block_sum(q[k], sh);
    if (threadIdx.x == 0) partials[(size_t)k * nb + bid] = b;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = (atomicAdd(ticket, 1u) == nb - 1) ? 1u : 0u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // last block: per-row sums in fixed order (thread t handles rows t, t+256, ...)
  double norm_part = 0.0, inside_part = 0.0, dip_part = 0.0;
  for (int row = threadIdx.x; row <= L; row += kObsThreads) {
    double p0 = 0.0, p1 = 0.0, p2 = 0.0;
    for (int bx = 0; bx < nbx; ++bx) {
      const size_t o = (size_t)row * nbx + bx;
      p0 += __ldcg(&partials[0 * nb + o]);
      p1 += __ldcg(&partials[1 * nb + o]);
      p2 += __ldcg(&partials[2 * nb + o]);
    }
    out[4 + row] = dr * p0;
    norm_part += p0;
    inside_part += p1;
    if (row < L) dip_part += 2.0 * kappa[row + 1] * dr * p2;
  }
  const double norm = block_sum(norm_part, sh);
  const double inside = block_sum(inside_part, sh);
  const double dip = block_sum(dip_part, sh);
  if (threadIdx.x == 0) {
    double ore = 0.0, oim = 0.0;
    for (int bx = 0; bx < nbx; ++bx) {
      ore += __ldcg(&partials[3 * nb + bx]);
      oim += __ldcg(&partials[4 * nb + bx]);
    }
    ore *= dr;
    oim *= dr;
    out[0] = dr * norm;
    out[1] = dip;
    out[2] = 1.0 - dr * inside;
    out[3] = ore * ore + oim * oim;
    *ticket = 0u;
  }
}

template <int WALK>
OpIn<WALK> make_in(const Geometry &g, const OperatorView &op, double E, const double2 *x) {
  OpIn<WALK> in;
  if constexpr (is_plain(WALK)) {
    in.diag = op.diag;
  } else {
    in.diagq = op.diagq;
    in.c1q = op.c1q;
    in.c2q = op.c2q;
    in.e1 = op.fx_e1;
    in.e2 = op.fx_e2;
    in.ec = op.fx_ec;
    in.ok = 1;
    in.k = 0;
  }
  in.rinv = op.rinv;
  in.d1c = (g.stencil == 5) ? 1.0 / (12.0 * g.dr) : 1.0 / (2.0 * g.dr);
  in.x = x;
  in.rj = op.rj;
  in.kappa = op.kappa;
  in.N = g.N;
  in.L = g.L;
  in.c1 = g.c1;
  in.c2 = g.c2;
  in.E = E;
  return in;
}

template <int V>
using IC = std::integral_constant<int, V>;
template <bool V>
using BC = std::integral_constant<bool, V>;

// f(stencil, walk) with both as compile-time constants.
template <typename F>
void dispatch(const Geometry &g, bool vg, bool plain, F &&f) {
  auto go = [&](auto st) {
    if (plain && vg) f(st, IC<kPlainVG>{});
    else if (plain) f(st, IC<kPlain>{});
    else if (vg) f(st, IC<kFixedVG>{});
    else f(st, IC<kFixed>{});
  };
  if (g.stencil == 5) go(IC<5>{});
  else go(IC<3>{});
}

// Persistent grids: a few blocks per SM (all resident at once).
template <int WALK>
inline unsigned stencil_blocks(const Geometry &g) { return (unsigned)(g.sms * kOpBlocksPerSM<WALK>); }
inline unsigned elem_blocks(const Geometry &g) { return (unsigned)(g.sms * kElemBlocksPerSM); }

// The parts a fixed-point launch's blocks are cut to: half the warps where the
// strips' row segments need no more.  Two blocks then fit on an SM, so that the
// next kernel of the chain is resident and waiting when this one ends.  The
// warps' numbers, and so every sum, stay the same.  (Lanczos-12, 17,600
// points: 312 to 267 us a step.)
inline unsigned block_parts(const Geometry &g) {
  const size_t per_sm = ((size_t)((g.N + kFxCols - 1) / kFxCols) * (g.L + 1) + g.sms - 1) / g.sms;
  return per_sm <= kBlockJ / 64 && (unsigned)g.sms <= kBlockJ / 2 ? 2u : 1u;
}

// A stencil kernel's launch: its rings are dynamic shared memory, raised above
// the 48 KB default once per instantiation and device.
template <auto KERN, int WALK, int EX>
OpLaunch op_launch(const Geometry &g) {
  constexpr size_t bytes = is_plain(WALK) ? 0 : (kBlockJ / 32) * (size_t)fx_warp_bytes<EX, WALK == kFixedVG>();
  static_assert(bytes <= 226 * 1024, "an SM's shared memory, less the kernel's own");
  const unsigned parts = is_plain(WALK) ? 1u : block_parts(g);
  if (!is_plain(WALK)) {
    // one split of L1 and shared memory for all of them: a kernel that wants
    // another than its predecessor's waits for the SM to drain (Dormand-Prince
    // on 50,000 points: 279 us for four steps, 233 with one split)
    const cudaError_t ready = kernel_ready<KERN>((int)bytes, cudaSharedmemCarveoutMaxShared);
    if (ready != cudaSuccess) return OpLaunch{0, 0, 0, ready};
  }
  return OpLaunch{stencil_blocks<WALK>(g), kBlockJ / parts, bytes / parts, cudaSuccess};
}

}  // namespace

// ---------------------------------------------------------------------------
cudaError_t launch_fx_diag(const double *diag, size_t G, int ec, long long *diagq, const Geometry &g, cudaStream_t s) {
  fx_diag_kernel<<<(unsigned)(g.sms * 4), 256, 0, s>>>(diag, G, ec, diagq);
  return cudaGetLastError();
}

cudaError_t launch_apply_h(const Geometry &g, const OperatorView &op, double E,
                           const double2 *x, double2 *y, cudaStream_t s) {
  cudaError_t e = cudaSuccess;
  dispatch(g, g.gauge == 1, op.plain, [&](auto st, auto walk) {
    constexpr int ST = decltype(st)::value;
    constexpr int WALK = decltype(walk)::value;
    const OpLaunch o = op_launch<apply_h_kernel<ST, WALK>, WALK, 0>(g);
    if ((e = o.ready) != cudaSuccess) return;
    apply_h_kernel<ST, WALK><<<o.grid, o.threads, o.bytes, s>>>(make_in<WALK>(g, op, E, x), y);
    e = cudaGetLastError();
  });
  return e;
}

cudaError_t launch_taylor_stage(const Geometry &g, const OperatorView &op, double E, double s,
                                const double2 *v_in, const double2 *psi, double2 *v_out,
                                bool final_stage, cudaStream_t st, bool imag) {
  const int mstart = op.mask_start;
  cudaError_t e = cudaSuccess;
  dispatch(g, !imag && g.gauge == 1, op.plain, [&](auto stc, auto walk) {
    constexpr int ST = decltype(stc)::value;
    constexpr int WALK = decltype(walk)::value;
    const auto in = make_in<WALK>(g, op, E, v_in);
    if constexpr (WALK == kFixed || WALK == kPlain)   // imaginary time: no absorber, no field
      if (imag) {
        e = launch_pdl(taylor_stage_kernel<ST, true, WALK, false>,
                       op_launch<taylor_stage_kernel<ST, true, WALK, false>, WALK, 1>(g), st, in, s, psi,
                       v_out, op.mask, mstart);
        return;
      }
    if (final_stage)
      e = launch_pdl(taylor_stage_kernel<ST, false, WALK, true>,
                     op_launch<taylor_stage_kernel<ST, false, WALK, true>, WALK, 1>(g), st, in, s, psi, v_out,
                     op.mask, mstart);
    else
      e = launch_pdl(taylor_stage_kernel<ST, false, WALK, false>,
                     op_launch<taylor_stage_kernel<ST, false, WALK, false>, WALK, 1>(g), st, in, s, psi, v_out,
                     op.mask, mstart);
  });
  return e;
}

cudaError_t launch_rk_stage(const Geometry &g, const OperatorView &op, double E, int stage,
                            double dt, const double2 *gin, const double2 *psi, double2 *acc,
                            double2 *g_next, double2 *psi_out, cudaStream_t st, bool imag) {
  // classic tableau: a_{s+1,s} = (1/2, 1/2, 1), b = (1, 2, 2, 1) / 6
  static const double a_next[4] = {0.5, 0.5, 1.0, 0.0};
  static const double b[4] = {1.0 / 6.0, 1.0 / 3.0, 1.0 / 3.0, 1.0 / 6.0};
  const double ca = dt * a_next[stage - 1], cb = dt * b[stage - 1];
  const int mstart = imag ? g.N : op.mask_start;
  cudaError_t e = cudaSuccess;
  dispatch(g, !imag && g.gauge == 1, op.plain, [&](auto stc, auto walk) {
    constexpr int ST = decltype(stc)::value;
    constexpr int WALK = decltype(walk)::value;
    const auto in = make_in<WALK>(g, op, E, gin);
    auto go = [&](auto part, auto im) {
      constexpr int PART = decltype(part)::value;
      constexpr bool IMAG = decltype(im)::value;
      constexpr int EX = PART == 0 ? 0 : (PART == 1 ? 2 : 1);
      e = launch_pdl(rk_stage_kernel<ST, IMAG, WALK, PART>,
                     op_launch<rk_stage_kernel<ST, IMAG, WALK, PART>, WALK, EX>(g), st, in, ca, cb, psi, acc, g_next,
                     psi_out, op.mask, mstart);
    };
    auto parts = [&](auto im) {
      if (stage == 1) go(IC<0>{}, im);
      else if (stage < 4) go(IC<1>{}, im);
      else go(IC<2>{}, im);
    };
    if constexpr (WALK == kFixed || WALK == kPlain)
      if (imag) return parts(BC<true>{});
    parts(BC<false>{});
  });
  return e;
}

cudaError_t launch_rk_general_stage(const Geometry &g, const OperatorView &op, double E,
                                    const double2 *gin, const double2 *psi, const RkStageArgs &a,
                                    Reduction *red, cudaStream_t st) {
  if (a.stage < 0 || a.stage >= kRkMaxStages) return cudaErrorInvalidValue;
  const double S = (double)g.N * (double)(g.L + 1);
  const int mode = a.last ? (a.fsal ? 2 : 1) : 0;
  cudaError_t e = cudaSuccess;
  if (!a.last && a.stage == kRkMaxStages - 1) return cudaErrorInvalidValue;   // no stage after the last
  if (a.fsal && (!a.last || a.stage == 0)) return cudaErrorInvalidValue;
  dispatch(g, g.gauge == 1, op.plain, [&](auto stc, auto walk) {
    constexpr int ST = decltype(stc)::value;
    constexpr int WALK = decltype(walk)::value;
    const auto in = make_in<WALK>(g, op, E, gin);
    auto launch = [&](auto nk, auto md) {
      constexpr int NK = decltype(nk)::value, MODE = decltype(md)::value;
      constexpr int VECS = MODE == 2 ? NK - 1 : NK, EX = VECS < 2 ? VECS : 2;
      e = launch_pdl(rk_general_stage_kernel<ST, WALK, NK, MODE>,
                     op_launch<rk_general_stage_kernel<ST, WALK, NK, MODE>, WALK, EX>(g), st, in, a, psi, op.mask,
                     op.mask_start, red, S);
    };
    auto go = [&](auto nk) {
      constexpr int NK = decltype(nk)::value;
      if (mode == 1) launch(nk, IC<1>{});
      if constexpr (NK > 1)
        if (mode == 2) launch(nk, IC<2>{});
      if constexpr (NK < kRkMaxStages)
        if (mode == 0) launch(nk, IC<0>{});
    };
    switch (a.stage + 1) {
      case 1: go(IC<1>{}); break;
      case 2: go(IC<2>{}); break;
      case 3: go(IC<3>{}); break;
      case 4: go(IC<4>{}); break;
      case 5: go(IC<5>{}); break;
      case 6: go(IC<6>{}); break;
      default: go(IC<7>{}); break;
    }
  });
  return e;
}

cudaError_t launch_imag_begin(const Reduction *red, double dr, double *imag_dev, cudaStream_t st) {
  imag_begin_kernel<<<1, 1, 0, st>>>(red, dr, imag_dev);
  return cudaGetLastError();
}

cudaError_t launch_imag_normalize(const Geometry &g, double2 *psi, const Reduction *red, double dt,
                                  double *imag_dev, cudaStream_t st) {
  const size_t G = (size_t)g.N * (g.L + 1);
  imag_normalize_kernel<<<elem_blocks(g), kElemThreads, 0, st>>>(G, psi, red, g.dr, dt, imag_dev);
  return cudaGetLastError();
}

cudaError_t launch_norm(const Geometry &g, const double2 *x, Reduction *red,
                        LanczosScalars *ls, int *status, cudaStream_t st) {
  const size_t G = (size_t)g.N * (g.L + 1);
  const cudaError_t e = launch_pdl(norm_kernel, elem_blocks(g), kElemThreads, 0, st, G, x, red, ls, status);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_lanczos_a(const Geometry &g, const OperatorView &op, double E, int j,
                             const double2 *u, const double2 *uprev, double2 *z,
                             Reduction *red, LanczosScalars *ls, cudaStream_t st) {
  cudaError_t e = cudaSuccess;
  dispatch(g, g.gauge == 1, op.plain, [&](auto stc, auto walk) {
    constexpr int ST = decltype(stc)::value;
    constexpr int WALK = decltype(walk)::value;
    const auto in = make_in<WALK>(g, op, E, u);
    if (j > 0) e = launch_pdl(lanczos_a_kernel<ST, WALK, 1>,
                   op_launch<lanczos_a_kernel<ST, WALK, 1>, WALK, 1>(g), st, in, j, uprev, z, red, ls);
    else e = launch_pdl(lanczos_a_kernel<ST, WALK, 0>,
                   op_launch<lanczos_a_kernel<ST, WALK, 0>, WALK, 0>(g), st, in, j, uprev, z, red, ls);
  });
  return e;
}

cudaError_t launch_lanczos_b(const Geometry &g, int j, const double2 *z, const double2 *u,
                             double2 *unext, Reduction *red, LanczosScalars *ls, cudaStream_t st) {
  const size_t G = (size_t)g.N * (g.L + 1);
  const cudaError_t e = launch_pdl(lanczos_b_kernel, elem_blocks(g), kElemThreads, 0, st, G, j, z, u, unext, red, ls);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_lanczos_combine(const Geometry &g, const OperatorView &op, int m,
                                   double2 *psi, const double2 *work, size_t stride,
                                   Reduction *red, LanczosScalars *ls, int *status,
                                   cudaStream_t st) {
  (void)m;
  const size_t G = (size_t)g.N * (g.L + 1);
  const cudaError_t e = launch_pdl(lanczos_combine_kernel, (unsigned)g.sms, kElemThreads, 0, st, G, g.N, psi, work,
                                   stride, op.mask, op.mask_start, red, ls, status);
  return e != cudaSuccess ? e : cudaGetLastError();
}

int observables_blocks(const Geometry &g) {
  const int per_row = (g.N + kObsThreads - 1) / kObsThreads;
  return per_row < 8 ? per_row : 8;
}

cudaError_t launch_observables(const Geometry &g, const OperatorView &op, const double2 *psi,
                               const double2 *ref0, double r_b, double *partials,
                               unsigned *ticket, double *out, cudaStream_t st) {
  const int nbx = observables_blocks(g);
  const dim3 grid(nbx, g.L + 1);
  observables_kernel<<<grid, kObsThreads, 0, st>>>(psi, ref0, op.rj, op.kappa, g.N, g.L, g.dr,
                                                   r_b, partials, ticket, out);
  return cudaGetLastError();
}

}  // namespace tdse_dev
