// Device helpers shared by the CUDA sources of libmolc.
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "molc_internal.h"

namespace molc {

// In a small step the kernels follow one another by programmatic dependent launch: a kernel calls chain_next at once, so
// that the next one's blocks are placed and load the plan's constants meanwhile, and chain_wait (until every earlier kernel
// of the chain has finished and its writes are visible) before they touch anything else.  The first kernel of a step is
// launched plainly: it starts after all earlier work of the stream, so nothing reaches back past it.  What an earlier kernel
// of the chain writes is read by ordinary loads after chain_wait, never through the read-only path (__ldg, ld.global.nc):
// that path takes its data to be constant while the kernel runs, and the wait orders ordinary loads only.
//
// A step is chained where its walks need no more blocks than there are SMs and the kernel ahead of its sweep is small too,
// link by link, from 240 shapes timed with each link on and off (times over those of plain launches):
//  - FP32, input preparation and moment gather: up to 4 blocks of the preparation an SM (0.78 to 1.00; beyond, 0.97 to 1.02).
//  - FP32, the sweep: it keeps the split of shared memory and L1 it finds on an SM for its whole, long run, and its blocks
//    go where the preparation leaves room, so this link pays only behind a preparation of at most one block an SM, and of
//    half of that where a sweep block has more shared memory than the preparation's (from 5 polar cosines).  With the
//    links above: 0.75 to 0.99; at 128 blocks of the preparation 0.91 with 4 polar cosines but 1.09 with 5 (0.97 without
//    this link), at 473 1.32 (0.96), at 1458 (216^2 cells, 1 group) 2.6.
//  - FP64: up to 48 blocks of the preparation (0.87 to 1.03); at 106 1.08, at 418 1.27.
// 16^2 x 4 groups: FP64 49.2 -> 43.1 us a step, FP32 26.6 -> 25.5.
inline bool few_walks(const PlanView &v) { return 2 * v.n_tracks * v.G <= 152 * kSweepBlock; }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... K, class... A>
cudaError_t launch_chained(bool chain, void (*kernel)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = chain ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
  if (e != cudaSuccess) cudaGetLastError();   // reported here, not by the next launch
  return e;
}

// Not (x >= 0 and finite), decided on the bits (integer pipe; the FP64 pipe is narrow): +0, -0 and the positive
// finite numbers pass.
__device__ __forceinline__ bool bad_input(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  return !(u < 0x7FF0000000000000ull || u == 0x8000000000000000ull);
}

// FP32 -> FP64 by integer operations (the FP64 conversion pipe is narrow on this GPU): exponent rebiased by
// 1023 - 127 and mantissa shifted into place, exact for normal numbers.  Zeros and subnormals (|x| < 2^-126)
// map to a value of the same sign and magnitude below 2^-126; the FP32 sweep works in units where max B is
// ~2^100, so that is below 1e-68 of max B.
__device__ __forceinline__ double f32_to_f64(float x) {
  const unsigned u = __float_as_uint(x);
  const unsigned hi = (u & 0x80000000u) | (((u >> 3) & 0x0fffffffu) + 0x38000000u);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// Exact FP32 -> FP64 for every finite x: the integer route for normal numbers, the conversion instruction for
// zeros and subnormals.
__device__ __forceinline__ double f32_to_f64_exact(float x) {
  return (__float_as_uint(x) & 0x7f800000u) ? f32_to_f64(x) : (double)x;
}

// Exponent k of a power of two x = 2^k (a normal double).
__device__ __forceinline__ int exponent_of(double x) { return ((__double2hiint(x) >> 20) & 0x7ff) - 1023; }

// x 2^k in FP64; by two products, as the factor itself may lie outside the normal range.  Out of line, so that the
// integer forms below, which call it for the few values they do not take, do not execute its FP64 operations for all.
static __device__ __noinline__ double scale_pow2_fp64(double x, int k) {
  const double h = __hiloint2double((1023 + (k >> 1)) << 20, 0), r = __hiloint2double((1023 + k - (k >> 1)) << 20, 0);
  return x * h * r;
}

// x 2^k as a double: integer operations where x is a normal float and the result a normal double, or x is zero.
__device__ __forceinline__ double scaled_to_double(float x, int k) {
  const unsigned u = __float_as_uint(x);
  const int e = (int)((u >> 23) & 0xff), ed = e - 127 + 1023 + k;
  if (e == 0 || e == 0xff || (unsigned)(ed - 1) >= 2046u) {
    if ((u << 1) == 0) return __hiloint2double((int)u, 0);
    return scale_pow2_fp64((double)x, k);
  }
  return __hiloint2double((int)((u & 0x80000000u) | ((unsigned)ed << 20) | ((u & 0x7fffffu) >> 3)), (int)(u << 29));
}

// x 2^k rounded to the nearest float (ties to even): integer operations where x and the float are normal, or x is zero.
__device__ __forceinline__ float scaled_to_float(double x, int k) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ff), ef = e - 1023 + k + 127;
  if (e == 0 || e == 0x7ff || (unsigned)(ef - 1) >= 253u) {
    if (((hi << 1) | lo) == 0) return __uint_as_float(hi);
    return (float)scale_pow2_fp64(x, k);
  }
  const unsigned f = ((hi & 0xfffffu) << 3) | (lo >> 29), rest = lo << 3;   // 23 bits, and what is cut
  return __uint_as_float((hi & 0x80000000u) | (((unsigned)ef << 23) + f + (rest > 0x80000000u - (f & 1))));
}

// What an FP32 sweep adds to the segment update: nothing, the face reductions of Eq. 16 (MOLC_FACES), or the
// per-ray balance check (MOLC_BALANCE).
enum SweepExtra { kSweepPlain = 0, kSweepFaces = 1, kSweepBalance = 2 };

// Per-ray balance (MOLC_BALANCE): R = I_in - I_out + sum_s tau_s (d_s - psibar_s), which is the integral of the
// transport equation along the characteristic, I_in - I_out + sum_s (Q_s - kappa~_s Ibar_s) l_s / sin zeta, in the
// deviation variables (Q - kappa~ Ibar = kappa~ (d - psibar)).  Segment by segment it reads
// I_in,s - I_out,s + tau_s (d_s - psibar_s) = 0, and the crossings add I_out,s - I_in,s+1 = 0 (the steps of B the
// deviation form takes there); S is the sum of the magnitudes of all these terms in the variables the sweep
// rounds (|I_in,s|, |I_out,s| and their deviations |psi_in,s|, |psi_out,s| from the cell's B, tau_s |B_s + d_s| =
// |Q_s| l_s / sin zeta, tau_s |B_s + psibar_s| = kappa~_s |Ibar_s| l_s / sin zeta, the B steps), so that |R| / S
// is a few units of the working precision's rounding when the arithmetic is consistent.  The largest |R| / S goes
// into *word by an integer atomicMax (non-negative doubles order like their bits).
// Rays whose terms sum to less than kBalanceFloor of max(B, boundary) (word[1], in the units of R and S after the
// factor `units`) carry no radiation at the working precision and are left out.
constexpr double kBalanceFloor = 1e-30;
__device__ __forceinline__ void ray_balance_max(unsigned long long *word, double R, double S, double units) {
  const double floor = kBalanceFloor * __longlong_as_double((long long)word[1]) * units;
  if (!(S > floor) || !(S > 0.0)) return;
  atomicMax(word, (unsigned long long)__double_as_longlong(fabs(R) / S));
}


// Eddington factors of one (cell, group) from the moments just assembled (Eq. 7 with the cell averages of
// Eq. 15): f = N / (c E), 0 where E = 0.  The same operations as closure_kernel, so molc_sweep_closure and
// molc_sweep + molc_closure give the same bits.
__device__ __forceinline__ void eddington_factors(const SweepArgs &a, int64_t idx, double E, double nxx, double nxy,
                                                  double nyy) {
  const double inv = E > 0 ? 1.0 / (a.c * E) : 0.0;
  a.fxx[idx] = nxx * inv;
  a.fxy[idx] = nxy * inv;
  a.fyy[idx] = nyy * inv;
}

// The FP64 sweep's cell entry; 1/(c dt kappa~) rounds like the quotient it replaces.
__device__ __forceinline__ Cell64 cell64(double kappa, double B, double Bref, double inv_cdt) {
  Cell64 c;
  c.kt = kappa + inv_cdt;
  c.r = inv_cdt / c.kt;
  c.B = B;
  c.dB = (Bref - B) * c.r;
  return c;
}

}  // namespace molc
