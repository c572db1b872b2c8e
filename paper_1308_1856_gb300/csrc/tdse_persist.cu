// Every Lanczos step of a tdse_propagate call in one cooperative launch (FP64,
// length gauge), for grids too large for one thread-block cluster.
//
// The multi-launch path (Appendix "Lanczos methods" of arXiv 1308.1856: per
// iteration j a stencil phase A, z = sigma_j H U_j - ratio_j U_{j-1} with
// alpha_j, and an elementwise phase B, U_{j+1} = z - alpha_j sigma_j U_j with
// beta_j; then the small exponential and the combine) issues 2m + 1 launches
// per step, and at 512,000 points each phase is a few microseconds of work
// behind a launch, a ramp and a grid reduction's tail.  Here the grid stays
// resident for the whole call and the phases are separated by a grid-wide
// barrier:
//   - the grid is the multi-launch stencil kernel's (one block of 512 threads
//     per SM), and every phase walks exactly the multi-launch kernel's work
//     split with the same arithmetic; in the elementwise phases, whose kernels
//     have kElemBlocksPerSM blocks an SM, a block stands for as many of them in turn;
//   - a reduction stores the block's partial, crosses the barrier, and then
//     EVERY block adds all partials in the multi-launch last block's fixed
//     order, so every block holds the same scalars and the results equal the
//     multi-launch path's bitwise;
//   - block 0 keeps the handle's Lanczos scalars in global memory up to date
//     and forms the small exponential in its first 256 threads (a named
//     barrier) while the other blocks wait at the next grid barrier;
//   - loads of anything another block wrote during the launch go to L2
//     (ld.global.cg): an SM's L1 is not kept coherent with other SMs' stores.
// The barrier waits are bounded: a block that polls more than kGridSpins
// times sets kStatusTimeout and carries on, so the launch always ends and the
// handle reports the error at its next synchronising call.  A cooperative
// launch is refused (not queued) when the grid cannot be resident at once.
#include <cuda_runtime.h>

#include "tdse_device_common.cuh"
#include "tdse_internal.cuh"
#include "tdse_small_expm.cuh"
#include "tdse_stencil.cuh"
#include "tdse_walk_fixed.cuh"
#include "tdse_combine_fixed.cuh"

namespace tdse_dev {
namespace {

using namespace common;
using namespace stencil;

constexpr long long kGridSpins = 1LL << 21;   // polls of the barrier's generation (~1 us each) before giving up
constexpr int kUnrollB = 4;                   // phase B: groups loaded before use (as the B kernel)

struct PersistArgs {
  FxIn in;                   // operator; x, k and E are set per phase
  double2 *psi;              // U_0, rewritten by the combine
  double2 *work;             // slot 0: z; slots 1..m-1: U_j
  size_t G;
  int m;
  double dt;
  long nsteps;
  const double *etab;        // coupling at each step's mid-point
  const double *mask;
  int mask_start;
  LanczosScalars *ls;
  Reduction *red;            // the handle's (normsq after each combine)
  Reduction *rp;             // two partial buffers, used in turn
  unsigned *bar;             // barrier: arrival count, generation
  int *status;
};

// Grid-wide barrier: every block's writes before it are visible (in L2) to
// every block after it.  Once any block has given up waiting (the status
// word's timeout bit), no block waits any more, so the launch ends quickly.
__device__ __forceinline__ void grid_sync(unsigned *bar, unsigned nblocks, int *status) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned *gen = bar + 1;
    volatile int *st = status;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(bar, 1u) == nblocks - 1u) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      long long spins = 0;
      while (*gen == g) {
        if (++spins > kGridSpins || (*st & kStatusTimeout)) {
          atomicOr(status, kStatusTimeout);
          break;
        }
        __nanosleep(32);
      }
    }
    __threadfence();
  }
  __syncthreads();
}

// The partials of the multi-launch blocks this block stands for (v[q]: block
// q gridDim + blockIdx of V gridDim blocks), the barrier, then every block's
// fixed-order sum of all partials (the multi-launch last block's reduce_partials).
template <int V>
__device__ __forceinline__ double grid_reduce(const double (&v)[V], Reduction *r, double *sh, const PersistArgs &a) {
#pragma unroll
  for (int q = 0; q < V; ++q) {
    const double b = block_sum(v[q], sh);
    if (threadIdx.x == 0) r->partial[q * gridDim.x + blockIdx.x] = b;
  }
  grid_sync(a.bar, gridDim.x, a.status);
  return reduce_partials(r, V * gridDim.x, sh);
}

// warp_range for multi-launch block q gridDim + blockIdx of V gridDim blocks.
template <int V>
__device__ __forceinline__ void elem_range(int q, long long total, long long &s0, long long &s1) {
  const unsigned nw = blockDim.x >> 5, W = V * gridDim.x * nw;
  const unsigned w = (q * gridDim.x + blockIdx.x) * nw + (threadIdx.x >> 5);
  const unsigned T = (unsigned)total, n = T / W, r = T - n * W;
  s0 = (long long)w * n + (w < r ? w : r);
  s1 = s0 + n + (w < r ? 1u : 0u);
}

template <int ST>
__global__ void __launch_bounds__(kBlockJ, 1) lanczos_persistent_kernel(PersistArgs a) {
  __shared__ double sh[kBlockJ / 32 + 1];
  __shared__ double s_sigma[kMaxKrylov + 1], s_ratio[kMaxKrylov + 1], s_acoef[kMaxKrylov];
  __shared__ double s_g[kMaxKrylov];   // step_scale's g_j
  __shared__ CbTable tab;
  extern __shared__ __align__(16) unsigned char fx_smem[];
  constexpr int V = kElemBlocksPerSM;
  static_assert(kElemThreads == kBlockJ, "a block stands for whole elementwise blocks");
  const int tid = threadIdx.x, lane = tid & 31;
  const bool lead = blockIdx.x == 0;
  const size_t G = a.G;
  int par = 0;
  if (tid == 0) s_sigma[0] = __ldcg(&a.ls->sigma[0]);
  __syncthreads();
  for (long n = 0; n < a.nsteps; ++n) {
    FxIn in = a.in;
    in.E = a.etab[n];
    for (int j = 0; j < a.m; ++j) {
      // ---- phase A (the lanczos_a kernel's arithmetic)
      const double sig = s_sigma[j];
      const StepScale sc = step_scale(sig);
      const double cprev = (j > 0) ? s_ratio[j] : 0.0;
      const double2 *u = (j == 0) ? a.psi : a.work + (size_t)j * G;
      double2 *z = a.work;
      in.x = u;
      in.k = sc.k;
      double acc[1] = {0.0};
      auto phase_a = [&](auto has_prev) {
        constexpr int EX = decltype(has_prev)::value;
        unsigned char *ring = fx_smem + (tid >> 5) * fx_warp_bytes<EX, false>();
        FxExtra<EX> ex;
        if (EX > 0) ex.p[0] = (j == 1) ? a.psi : a.work + (size_t)(j - 1) * G;
        for_my_strips(in, [&](int j0, int l0, int l1) {
          walk_rows_fixed<ST, false, EX>(in, ex, ring, j0, l0, l1,
                                  [&](int idx, int, double2 t, double2 uu, const double2 (&e)[1]) {
            double2 o = t;
            if (EX > 0) {
              o.x = __fma_rn(-cprev, e[0].x, t.x);
              o.y = __fma_rn(-cprev, e[0].y, t.y);
            }
            z[idx] = o;
            acc[0] = __fma_rn(uu.x, o.x, acc[0]);
            acc[0] = __fma_rn(uu.y, o.y, acc[0]);
          });
        });
      };
      if (j > 0) phase_a(std::integral_constant<int, 1>{});
      else phase_a(std::integral_constant<int, 0>{});
      const double sa = grid_reduce(acc, a.rp + par, sh, a);
      par ^= 1;
      if (tid == 0) {
        const double al = (sa * sig) * sc.g;   // store_alpha
        s_acoef[j] = -al * sc.s;
        s_g[j] = sc.g;
        if (lead) {
          a.ls->alpha[j] = al;
          a.ls->acoef[j] = -al * sc.s;
        }
      }
      __syncthreads();
      if (j + 1 >= a.m) break;
      // ---- phase B (the lanczos_b kernel's arithmetic and work split)
      const double c = s_acoef[j];
      double2 *un = a.work + (size_t)(j + 1) * G;
      double accb[V];
#pragma unroll 1
      for (int q = 0; q < V; ++q) {
        double acc0 = 0.0, acc1 = 0.0;
        long long g0, g1;
        elem_range<V>(q, (long long)((G + 31) >> 5), g0, g1);
        for (long long gb = g0; gb < g1; gb += kUnrollB) {
          double2 zz[kUnrollB], vv[kUnrollB];
#pragma unroll
          for (int r = 0; r < kUnrollB; ++r) {
            const size_t idx = (size_t)(gb + r) * 32 + lane;
            const bool ok = (gb + r < g1) && idx < G;
            zz[r] = ok ? __ldcg(z + idx) : make_double2(0.0, 0.0);
            vv[r] = ok ? __ldcg(u + idx) : make_double2(0.0, 0.0);
          }
#pragma unroll
          for (int r = 0; r < kUnrollB; ++r) {
            const size_t idx = (size_t)(gb + r) * 32 + lane;
            if ((gb + r < g1) && idx < G) {
              const double2 o = make_double2(__fma_rn(c, vv[r].x, zz[r].x), __fma_rn(c, vv[r].y, zz[r].y));
              un[idx] = o;
              acc0 = __fma_rn(o.x, o.x, acc0);
              acc1 = __fma_rn(o.y, o.y, acc1);
            }
          }
        }
        accb[q] = acc0 + acc1;
      }
      const double sb = grid_reduce(accb, a.rp + par, sh, a);
      par ^= 1;
      if (tid == 0) {
        double nrm, sn;                        // store_beta
        norm_and_inverse(sb, nrm, sn);
        const double beta = s_g[j] * nrm;
        const double ratio = (sn > 0.0) ? (s_sigma[j] * beta) * (nrm * step_scale(sn).s) : 0.0;
        s_sigma[j + 1] = sn;
        s_ratio[j + 1] = ratio;
        if (lead) {
          a.ls->beta[j] = beta;
          a.ls->sigma[j + 1] = sn;
          a.ls->ratio[j + 1] = ratio;
        }
      }
      __syncthreads();
    }
    // ---- the small exponential: block 0's first kEx threads
    if (lead && tid < kEx) expm_body(a.m, a.dt, a.ls, false, ExNamedSync{});
    grid_sync(a.bar, gridDim.x, a.status);
    if (tid < 32) cb_setup(tab, a.ls);
    __syncthreads();
    // ---- the combine (the lanczos_combine kernel's arithmetic and work split)
    const int N = a.in.N;
    const double2 *U1 = a.work + G;
    double accn[1] = {0.0};
    {
      long long g0, g1;
      elem_range<1>(0, (long long)((G + 31) >> 5), g0, g1);
      for (long long gi = g0; gi < g1; ++gi) {
        const size_t idx = (size_t)gi * 32 + lane;
        const bool ok = idx < G;
        double2 o = cb_sum(tab, [&](int j) {
          return ok ? __ldcg(j == 0 ? a.psi + idx : U1 + (size_t)(j - 1) * G + idx) : make_double2(0.0, 0.0);
        });
        if (!ok) continue;
        const int jr = (int)((unsigned)idx % (unsigned)N);
        if (jr >= a.mask_start) {
          const double mv = a.mask[jr];
          o.x = __dmul_rn(mv, o.x);
          o.y = __dmul_rn(mv, o.y);
        }
        a.psi[idx] = o;
        accn[0] = __fma_rn(o.x, o.x, accn[0]);
        accn[0] = __fma_rn(o.y, o.y, accn[0]);
      }
    }
    const double sn2 = grid_reduce(accn, a.rp + par, sh, a);
    par ^= 1;
    if (tid == 0) {
      double nrm;
      norm_and_inverse(sn2, nrm, s_sigma[0]);
      if (lead) {
        a.red->normsq = sn2;
        a.ls->psinorm = nrm;
        a.ls->sigma[0] = s_sigma[0];
        if (!isfinite(sn2)) atomicOr(a.status, kStatusNonFinite);
      }
    }
    __syncthreads();
  }
}

}  // namespace

constexpr int kPersistSmem = (kBlockJ / 32) * fx_warp_bytes<1, false>();

bool lanczos_persistent_fits(int stencil) {
  int dev = 0, coop = 0, nb = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return false;
  }
  auto *kern = (stencil == 5) ? lanczos_persistent_kernel<5> : lanczos_persistent_kernel<3>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPersistSmem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, kBlockJ, kPersistSmem);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return nb >= 1;
}

size_t lanczos_persistent_scratch_bytes() { return 2 * sizeof(Reduction) + 2 * sizeof(unsigned); }

cudaError_t launch_lanczos_persistent(const Geometry &g, const OperatorView &op, int m, double dt, long nsteps,
                                      const double *etab, double2 *psi, double2 *work, LanczosScalars *ls,
                                      Reduction *red, void *scratch, int *status, cudaStream_t st) {
  PersistArgs a;
  FxIn &in = a.in;
  in.x = psi;
  in.diagq = op.diagq;
  in.rj = op.rj;
  in.kappa = op.kappa;
  in.N = g.N;
  in.L = g.L;
  in.c1 = g.c1;
  in.c2 = g.c2;
  in.c1q = op.c1q;
  in.c2q = op.c2q;
  in.e1 = op.fx_e1;
  in.e2 = op.fx_e2;
  in.ec = op.fx_ec;
  in.ok = 1;
  in.k = 0;
  in.E = 0.0;
  in.rinv = nullptr;
  in.d1c = 0.0;
  a.psi = psi;
  a.work = work;
  a.G = (size_t)g.N * (g.L + 1);
  a.m = m;
  a.dt = dt;
  a.nsteps = nsteps;
  a.etab = etab;
  a.mask = op.mask;
  a.mask_start = op.mask_start;
  a.ls = ls;
  a.red = red;
  a.rp = static_cast<Reduction *>(scratch);
  a.bar = reinterpret_cast<unsigned *>(static_cast<char *>(scratch) + 2 * sizeof(Reduction));
  a.status = status;
  cudaError_t e = cudaMemsetAsync(a.bar, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)g.sms, 1, 1);
  cfg.blockDim = dim3(kBlockJ, 1, 1);
  cfg.dynamicSmemBytes = kPersistSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (g.stencil == 5) return cudaLaunchKernelEx(&cfg, lanczos_persistent_kernel<5>, a);
  return cudaLaunchKernelEx(&cfg, lanczos_persistent_kernel<3>, a);
}

}  // namespace tdse_dev
