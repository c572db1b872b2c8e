// Device helpers shared by the FP64 and mixed-precision kernels: the
// persistent-grid work split and the deterministic grid reductions.
#pragma once

#include <cuda_runtime.h>

#include "tdse_fixed.cuh"
#include "tdse_internal.cuh"

namespace tdse_dev {
namespace common {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The warp's sum in fixed point (tdse_fixed.cuh: fx_addend, fx_total): integers
// against the largest exponent, added by the warp reduction instructions.  One
// FP64 instruction instead of five dependent ones of 64 cycles, which all warps
// of an SM sub-partition queue for: the tail of every reduction.  The sum is the
// same in any order, and its rounding is below the tree's.  A warp with an Inf
// or NaN, and sums at FP64's limits, take the tree.  Lanczos-12 on 512,000
// points, with the last block's sum of one partial a thread: 465 to 378 us a step in
// FP64, 295 to 200 mixed.
__device__ __forceinline__ double warp_sum_fx(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
  const unsigned e = __reduce_max_sync(0xffffffffu, (hi & tdse_fx::kExpMask) >> 20);
  if (e < tdse_fx::kSumLo || e > tdse_fx::kSumHi)
    return __any_sync(0xffffffffu, ((hi << 1) | lo) != 0) ? warp_sum(v) : 0.0;
  const int64_t X = tdse_fx::fx_addend(hi, lo, (int)e);
  const unsigned p0 = __reduce_add_sync(0xffffffffu, (unsigned)X & 0xfffffu);
  const unsigned p1 = __reduce_add_sync(0xffffffffu, (unsigned)(X >> 20) & 0xfffffu);
  const int p2 = __reduce_add_sync(0xffffffffu, (int)(X >> 40));
  const double t = __ll2double_rn(tdse_fx::fx_total(p0, p1, p2));
  const int h = __double2hiint(t);
  return __hiloint2double(h ? h + (((int)e - tdse_fx::kSumBias) << 20) : 0, __double2loint(t));
}

// Deterministic block sum (warp sums, then the sum of those); the result
// is valid in every thread.  `sh` needs blockDim/32 + 1 doubles.
__device__ __forceinline__ double block_sum(double v, double *sh) {
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  const int nthreads = blockDim.x * blockDim.y;
  v = warp_sum_fx(v);
  if ((tid & 31) == 0) sh[tid >> 5] = v;
  __syncthreads();
  if (tid < 32) {
    const int nw = nthreads >> 5;
    const double s = warp_sum_fx((tid < nw) ? sh[tid] : 0.0);
    if (tid == 0) sh[nw] = s;
  }
  __syncthreads();
  const double r = sh[nthreads >> 5];
  __syncthreads();
  return r;
}

// Called by every thread of the last block: fixed-order sum of all partials.
// Up to one partial a thread (every grid of the library): the block sum alone.
// More: each thread first issues all its loads (independent, so their latencies
// overlap) and then adds them in index order.
constexpr int kMaxPartialsPerThread = 16;
__device__ __forceinline__ double reduce_partials(Reduction *red, unsigned nparts, double *sh) {
  const int tid = threadIdx.x + threadIdx.y * blockDim.x;
  const int nthreads = blockDim.x * blockDim.y;
  __threadfence();
  if (nparts <= (unsigned)nthreads) {
    const double t = block_sum((unsigned)tid < nparts ? __ldcg(&red->partial[tid]) : 0.0, sh);
    if (tid == 0) red->ticket = 0u;
    return t;
  }
  double v[kMaxPartialsPerThread];
#pragma unroll
  for (int r = 0; r < kMaxPartialsPerThread; ++r) {
    const unsigned k = tid + (unsigned)r * nthreads;
    v[r] = (k < nparts) ? __ldcg(&red->partial[k]) : 0.0;
  }
  double s = 0.0;
#pragma unroll
  for (int r = 0; r < kMaxPartialsPerThread; ++r) s += v[r];
  s = block_sum(s, sh);
  if (tid == 0) red->ticket = 0u;
  return s;
}

// Global warp index and warp count of a 1-D persistent launch.
// Running sum of FP32 terms held as an unevaluated pair s + c: every addition
// is error-free (Knuth's TwoSum), so the pair keeps about twice the FP32
// precision and a long run of terms needs no FP64 arithmetic until value().
// (FP64 instructions, conversions included, issue at a small fraction of the
// FP32 rate on this part.)
struct PairSum {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float t = __fadd_rn(s, x);
    const float z = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z)));
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

__device__ __forceinline__ int warp_id() { return blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); }
__device__ __forceinline__ int warp_count() { return gridDim.x * (blockDim.x >> 5); }

// Range [s0, s1) of `total` (< 2^32) work items owned by warp w of the W warps:
// q = total / W items each, one more for the first total - q W warps.  Only a
// 32-bit division: a 64-bit integer division compiles to FP64 arithmetic,
// which issues at 1/64 of the FP32 rate on this part.
__device__ __forceinline__ void warp_range(long long total, long long &s0, long long &s1) {
  const unsigned W = (unsigned)warp_count(), w = (unsigned)warp_id();
  const unsigned T = (unsigned)total;
  const unsigned q = T / W, r = T - q * W;
  s0 = (long long)w * q + (w < r ? w : r);
  s1 = s0 + q + (w < r ? 1u : 0u);
}

// Sum v over the block (as block_sum), store it as this
// block's partial and report whether this block is the last to finish.  The
// last block then adds all block partials in a fixed order, so the result does
// not depend on timing.
__device__ __forceinline__ bool publish_block_partial(double v, Reduction *red, double *sh) {
  __shared__ unsigned s_last;
  v = warp_sum_fx(v);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {   // block_sum's sum, where it is needed
    const double b = warp_sum_fx(threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0);
    if (threadIdx.x == 0) {
      red->partial[blockIdx.x] = b;
      __threadfence();
      const unsigned t = atomicAdd(&red->ticket, 1u);
      s_last = (t == gridDim.x - 1) ? 1u : 0u;
    }
  }
  __syncthreads();
  return s_last != 0;
}

// ||x|| and 1 / ||x|| from ||x||^2 with one reciprocal square root, corrected to
// the nearest doubles (tdse_fixed.cuh: fx_norm).  Of a Lanczos-12 step's 376 us the
// corrections take 4; a square root and a division take more (each ~650 cycles).
// 0 gives (0, 0), Inf or NaN gives (sqrt, 0).
__device__ __forceinline__ void norm_and_inverse(double s2, double &nrm, double &inv) {
  if (s2 > 1e-280 && s2 <= 1.7976931348623157e308) {
    tdse_fx::fx_norm(s2, rsqrt(s2), nrm, inv);
  } else {
    nrm = sqrt(s2);
    inv = nrm > 0.0 ? 1.0 / nrm : 0.0;
  }
}

// The scale of the FP64 Lanczos recurrence.  z = s_j H U_j - ratio_j U_{j-1} with
// s_j the power of two at or below sigma_j (the scale is then an exponent, not
// a product per point) and ratio_j = beta_{j-1} sigma_{j-1} / g_j; with
// g_j = sigma_j / s_j in [1, 2):
//   alpha_j = sigma_j g_j Re<U_j, z>,  U_{j+1} = z - alpha_j s_j U_j,
//   beta_j = g_j ||U_{j+1}||.
// sigma_j = 0 (a vanished vector) keeps s_j = 1, g_j = 0.
struct StepScale {
  double s, g;
  int k;       // s = 2^k
};
__device__ __forceinline__ StepScale step_scale(double sigma) {
  StepScale r;
  const int f = (__double2hiint(sigma) >> 20) & 0x7ff;
  const bool usable = f > 0 && f < 0x7ff;
  r.k = usable ? f - 1023 : 0;
  r.s = usable ? __hiloint2double(f << 20, 0) : 1.0;
  r.g = usable ? __hiloint2double((__double2hiint(sigma) & 0xfffff) | 0x3ff00000, __double2loint(sigma)) : sigma;
  return r;
}

// alpha_j and U_{j+1}'s coefficient from the sum of U_j^* z.
__device__ __forceinline__ void store_alpha(LanczosScalars *ls, int j, double sum) {
  const double sig = ls->sigma[j];
  const StepScale sc = step_scale(sig);
  const double al = (sum * sig) * sc.g;
  ls->alpha[j] = al;
  ls->acoef[j] = -al * sc.s;
}
// beta_j and the next vector's scalars from ||U_{j+1}||^2.
__device__ __forceinline__ void store_beta(LanczosScalars *ls, int j, double sumsq) {
  double nrm, sn;
  norm_and_inverse(sumsq, nrm, sn);
  const double beta = step_scale(ls->sigma[j]).g * nrm;
  ls->beta[j] = beta;
  ls->sigma[j + 1] = sn;
  // 1 / g_{j+1} = s_{j+1} ||U_{j+1}||.  Formed here, in one thread: as a division in every
  // warp of the next kernel it took 2 us of that kernel
  ls->ratio[j + 1] = (sn > 0.0) ? (ls->sigma[j] * beta) * (nrm * step_scale(sn).s) : 0.0;
}

}  // namespace common
}  // namespace tdse_dev
