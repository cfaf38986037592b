// The plain FP64 sweep (MOLC_FP64) of libmolc on sm_103a.
//
// What bounds it: this GPU's FP64 pipe issues about 2 lanes per clock and SM (1.25e12 FLOP/s measured by
// molc_fp64_fma_rate), so one FP64 instruction of a warp takes 16 clocks of an SM in which its schedulers can issue 64
// other warp-instructions.  One thread therefore walks a (track, sense, group) with up to 8 polar cosines and keeps in
// FP64 only what carries the intensity (five operations an update: the crossing step, d, psi - d, psibar, psi) and the
// polar folds of the moments (three); per segment and group one product kappa~ l, one crossing difference, eight
// products and six atomics are shared by its polar cosines.  The attenuation (Eqs. 12-13), two transcendental
// functions and two divisions an update when taken in FP64, is evaluated on the integer pipe in 64-bit fixed point.
// 128^2 cells, 17 groups, 8 x 64 directions, h/2 (3.64e8 updates): 48.3 ms with FP64 exp, expm1, two divisions and six
// atomics an update on one thread per polar cosine; 7.7 ms so, of which about ten FP64
// operations an update take 5.8 ms at the measured rate.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "molc_device.cuh"
#include "molc_internal.h"

namespace molc {

namespace {

using u64 = unsigned long long;
using u32 = unsigned int;

// 2^(-j/64) in units of 2^-63, rounded to nearest (the table of a table-driven exponential in the manner of
// P. T. P. Tang, ACM TOMS 15 (1989) 144, with a power series in the remainder).
__constant__ u64 kExp2Table[64] = {
    0x8000000000000000ull, 0x7e9f06067a4360baull, 0x7d41d96db915019dull, 0x7be86fb985689ddcull,
    0x7a92be8a92436616ull, 0x7940bb9e2cffd89dull, 0x77f25ccdee6d7ae6ull, 0x76a7980f6cca15c2ull,
    0x75606373ee921c97ull, 0x741cb5281e25ee34ull, 0x72dc8373be41a454ull, 0x719fc4b95f452d29ull,
    0x70666f76154a7089ull, 0x6f307a412f074892ull, 0x6dfddbcbed791babull, 0x6cce8ae13c57ebdbull,
    0x6ba27e656b4eb57aull, 0x6a79ad55e7f6fd10ull, 0x69540ec8f895722dull, 0x683199ed779592caull,
    0x6712460a8fc24072ull, 0x65f60a7f79393e2eull, 0x64dcdec3371793d1ull, 0x63c6ba6455dcd8aeull,
    0x62b39508aa836d6full, 0x61a3666d124bb204ull, 0x6096266533384a2bull, 0x5f8bccdb3d398841ull,
    0x5e8451cfac061b5full, 0x5d7fad59099f22feull, 0x5c7dd7a3b17dcf75ull, 0x5b7ec8f19468bbc9ull,
    0x5a827999fcef3242ull, 0x5988e20954889245ull, 0x5891fac0e95612c8ull, 0x579dbc56b48521baull,
    0x56ac1f752150a563ull, 0x55bd1cdad49f699cull, 0x54d0ad5a753e077cull, 0x53e6c9da74b29ab5ull,
    0x52ff6b54d8a89c75ull, 0x521a8ad704f3404full, 0x513821818624b40cull, 0x50582887dcb8a7e1ull,
    0x4f7a993048d088d7ull, 0x4e9f6cd3967fdba8ull, 0x4dc69cdceaa72a9cull, 0x4cf022c9905bfd32ull,
    0x4c1bf828c6dc54b8ull, 0x4b4a169b900c2d00ull, 0x4a7a77d47f7b84b1ull, 0x49ad159789f37496ull,
    0x48e1e9b9d588e19bull, 0x4818ee218a3358eeull, 0x47521cc5a2e6a9e0ull, 0x468d6fadbf2dd4f3ull,
    0x45cae0f1f545eb73ull, 0x450a6abaa4b77ecdull, 0x444c0740496d4294ull, 0x438fb0cb4f468808ull,
    0x42d561b3e6243d8aull, 0x421d1461d66f2023ull, 0x4166c34c5615d0ecull, 0x40b268f9de0183baull,
};

// High 64 bits of a 64 x 64-bit product without the carries of its low half: at most 3 units too small.
__device__ __forceinline__ u64 mulhi(u64 a, u64 b) {
  const u32 a0 = (u32)a, a1 = (u32)(a >> 32), b0 = (u32)b, b1 = (u32)(b >> 32);
  return (u64)a1 * b1 + (u64)__umulhi(a1, b0) + (u64)__umulhi(a0, b1);
}

// P 2^e as a double, rounded to nearest (halves up); P normalised (top bit set).  The first form takes results in the
// normal range; the second also those below it, down to zero.
__device__ __forceinline__ double fixed_to_double(u64 P, int e) {
  const u64 m = (P >> 11) + ((P >> 10) & 1);
  return __longlong_as_double((long long)(m + ((u64)(u32)(e + 1085) << 52)));
}

__device__ __forceinline__ double fixed_to_small_double(u64 P, int e) {
  const u64 m = (P >> 11) + ((P >> 10) & 1);
  return __longlong_as_double((long long)((m >> min(max(-1085 - e, 0), 63)) + ((u64)(u32)max(e + 1085, 0) << 52)));
}

// A positive normal double as M 2^(e - 63), M normalised.
__device__ __forceinline__ u64 double_mantissa(double x, int &e) {
  const u64 b = (u64)__double_as_longlong(x);
  e = (int)(b >> 52) - 1023;
  return (b << 11) | 0x8000000000000000ull;
}

// 2^64 / m for m = M 2^-63 in [1, 2): the FP32 reciprocal of m's leading bits and one step of the third-order
// iteration y (1 + e + e^2), e = 1 - m y, |e| < 2^-21, all in fixed point (error below 2^-61 relative).
__device__ __forceinline__ u64 fixed_reciprocal(u64 M) {
  const float mf = __uint_as_float(0x3f800000u | ((u32)(M >> 40) & 0x7fffffu));
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(mf));
  // yf in (1/2, 1] to 32 fraction bits; 1 (and anything rounded above it) becomes 1 - 2^-32
  const u32 yb = max(__float_as_uint(yf), 0x3f000000u);
  const u32 Y = yb >= 0x3f800000u ? 0xffffffffu : ((yb << 8) | 0x80000000u);
  const u64 t = (u64)(u32)(M >> 32) * Y + (u64)__umulhi((u32)M, Y);       // m y 2^63
  const long long d = (long long)(t - 0x8000000000000000ull);              // -e 2^63
  const int ds = (int)(d >> 11);                                           // -e 2^52
  const long long corr = (((long long)ds * ds) >> 41) - d;                 // (e + e^2) 2^63
  const long long r = (long long)(int)(corr >> 32) * (long long)Y * 2 + (long long)(((u64)(u32)corr * Y) >> 31);
  const u64 y = ((u64)Y << 32) + (u64)r;
  return y >> 62 ? y : ~0ull;   // 1 itself (m = 1) wraps to 0
}

// E1 = (1 - e^-tau)/tau and, of the outgoing intensity's two forms, thin (tau < 1/2): f = 1 - e^-tau, else f = e^-tau,
// for tau = kl / sin zeta with kl = Mk 2^(ek - 63) and 1/kl = Mr 2^(-ek - 64).  z = tau log2 e is split into n + j/64 +
// u / ln 2 with 0 <= u < ln 2 / 64, and phi(u) = (1 - e^-u)/u = sum (-u)^k / (k + 1)! (truncated after u^6: below
// 2^-61 of it), so that e^-tau = 2^-n 2^(-j/64) (1 - u phi(u)).  For n = j = 0, u is tau and phi is E1 itself, which
// keeps the relative accuracy of 1 - e^-tau = tau E1 down to tau = 0; elsewhere 1 - e^-tau > 0.01 is formed from the
// fixed-point e^-tau (2^-63 absolute).  Products with the 64-bit mantissas of 1/sin zeta, sin zeta and
// log2 e / sin zeta stand for the FP64 products and divisions, each result being rounded to FP64 once (worst relative
// errors found over tau in [1e-12, 700] against 200-bit arithmetic: 2^-53 times 1.1 in f for tau < 1/2, 1.5 in E1).
__device__ __forceinline__ void attenuation_fixed(u64 Mk, int ek, u64 Mr, const PolarFix &c, const u64 *table,
                                                  double &E1, double &f, bool &thin) {
  u64 h = mulhi(Mk, c.Mz) >> 4;          // z 2^(58 - exponent)
  const int sh = ek + c.ez + 6;
  h >>= min(max(-sh, 0), 63);
  const int sl = min(max(sh, 0), 20);    // beyond 2^14 (e^-tau = 0) z only has to stay large
  const u32 n = __funnelshift_l((u32)(h >> 32), 0u, sl);
  const u64 F = h << sl;                 // fraction of z
  const u32 j = (u32)(F >> 58);
  const u64 U = __umul64hi(F & 0x03ffffffffffffffull, 0xb17217f7d1cf79acull);   // u 2^64 (ln 2)
  const u32 uh = (u32)(U >> 26);         // u 2^38
  const u32 b6 = 5965232u - __umulhi(uh, 13315u);                  // 1/720 - u/5040, 2^32
  const u32 b5 = 2290649225u - __umulhi(uh, b6);                   // 1/120 - u b6, 2^38
  const u64 b4 = 0x0aaaaaaaaaaaaaaaull - (((u64)uh * b5) >> 12);   // 1/24 - u b5, 2^64
  const u64 b3 = 0x2aaaaaaaaaaaaaaaull - mulhi(U, b4);             // 1/6 - u b4
  const u64 b2 = 0x8000000000000000ull - mulhi(U, b3);             // 1/2 - u b3
  const u64 phi = ~mulhi(U, b2);                                   // 1 - u b2 (less 2^-64)
  const u64 t = table[j];
  const u64 res = t - mulhi(t, mulhi(U, phi));                     // e^-tau 2^(n + 63)
  const bool first = (n | j) == 0;
  thin = n == 0 && (u32)(F >> 32) < 0xb8aa3b29u;                   // z < log2(e) / 2
  const u64 om = 0x8000000000000000ull - (res >> min(n, 63u));     // (1 - e^-tau) 2^63
  const int lz = __clz((int)(om >> 32));
  const u64 omn = om << lz;
  // first: 1 - e^-tau = tau phi; else E1 = (1 - e^-tau)/tau
  const u64 x = mulhi(first ? Mk : Mr, first ? c.Mi : c.Ms);
  u64 P = mulhi(x, first ? phi : omn);
  const int cp = __clz((int)(P >> 32));
  const double prod = fixed_to_double(P << cp, (first ? ek + c.ei - 62 : c.es - ek - lz - 62) - cp);
  // first: E1 = phi; else the factor of the outgoing intensity
  const int cr = __clz((int)(res >> 32));
  const u64 q = first ? phi : thin ? omn : res << cr;
  const int eq = first ? -64 : thin ? -63 - lz : -63 - cr - (int)n;
  const double other = fixed_to_small_double(q, eq);
  E1 = first ? other : prod;
  f = first ? prod : other;
}

// The same in FP64, for kappa~ l outside [2^-900, 2^900] (not a finite normal number of ordinary size).
__device__ __noinline__ void attenuation_fp64(double tau, double &E1, double &f, bool &thin) {
  const double om = -expm1(-tau);
  E1 = om / tau;
  thin = tau < 0.5;
  f = thin ? om : exp(-tau);
}

// The part of a polar cosine's constants that the attenuation reads.
__device__ __forceinline__ PolarFix load_polar(const PolarFix *p) {
  const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(p);
  const ulonglong2 a = __ldg(q), b = __ldg(q + 1);
  PolarFix r;
  r.Mz = a.x;
  r.Mi = a.y;
  r.Ms = b.x;
  r.ez = (int)(short)b.y;
  r.ei = (int)(short)(b.y >> 16);
  r.es = (int)(short)(b.y >> 32);
  return r;
}

// Input checks, cell entries and cleared accumulators; one thread per (group, cell), cells fastest (an entry is one
// 32-byte sector, the accumulators are cleared in memory order).
__global__ void __launch_bounds__(256) prep_fp64_kernel(PlanView v, SweepArgs a) {
  chain_next();
  const int64_t n = (int64_t)v.G * v.ncell, stride = (int64_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const double kap = a.kappa[i], B = a.B[i];
    bad |= bad_input(kap) | bad_input(B);
    if (a.cell64) {
      const int g = (int)(i / v.ncell), cell = (int)(i - (int64_t)g * v.ncell);
      a.cell64[(int64_t)cell * v.G + g] = cell64(kap, B, a.Bref[i], a.inv_cdt);
    }
#pragma unroll
    for (int o = 0; o < kOutputs; ++o) a.acc[o * n + i] = 0.0;
  }
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < 4 * v.G; i += blockDim.x) bad |= bad_input(a.bnd[i]);
  if (bad) atomicOr(v.status, kStatusNonfinite);
}

// Cell assembly.  acc holds sum_m omega_m sum_{C(i,m)} (A/V) psibar (times Omega components); the B_i part uses the
// geometric moments geo = sum_m omega_m sum_{C(i,m)} A/V (times Omega components):
//   E = (B geo0 + D)/c, F = acc, N_ab = B geo_ab + acc_ab   (the B part of F is zero by symmetry), and B_ref := B.
// A block turns 32 cells x 8 groups of [cell][6][G] accumulators into [g][cell] outputs through shared memory.
constexpr int kFinalCells = 32, kFinalGroups = 8;
__global__ void __launch_bounds__(kFinalCells *kFinalGroups) finalize_fp64_kernel(PlanView v, SweepArgs a) {
  __shared__ double sm[kOutputs][kFinalGroups][kFinalCells + 1];
  chain_wait();
  const int c0 = blockIdx.x * kFinalCells, g0 = blockIdx.y * kFinalGroups;
  const int nc = min(kFinalCells, v.ncell - c0), ng = min(kFinalGroups, v.G - g0);
  for (int k = threadIdx.x; k < nc * kOutputs * kFinalGroups; k += blockDim.x) {
    const int gl = k % kFinalGroups, co = k / kFinalGroups, o = co % kOutputs, cl = co / kOutputs;
    if (gl < ng) sm[o][gl][cl] = a.acc[((int64_t)(c0 + cl) * kOutputs + o) * v.G + g0 + gl];
  }
  __syncthreads();
  const int cl = threadIdx.x % kFinalCells, gl = threadIdx.x / kFinalCells;
  if (cl >= nc || gl >= ng) return;
  const int cell = c0 + cl;
  const int64_t idx = (int64_t)(g0 + gl) * v.ncell + cell;
  const double is = a.scale[1];   // 1 for an FP64 state
  const double B = a.B[idx];
  const double E = (B * v.geo[cell] + sm[0][gl][cl] * is) * a.inv_c;
  const double nxx = B * v.geo[v.ncell + cell] + sm[3][gl][cl] * is;
  const double nxy = B * v.geo[2 * (int64_t)v.ncell + cell] + sm[4][gl][cl] * is;
  const double nyy = B * v.geo[3 * (int64_t)v.ncell + cell] + sm[5][gl][cl] * is;
  a.out.E[idx] = E;
  a.out.Fx[idx] = sm[1][gl][cl] * is;
  a.out.Fy[idx] = sm[2][gl][cl] * is;
  a.out.Nxx[idx] = nxx;
  a.out.Nxy[idx] = nxy;
  a.out.Nyy[idx] = nyy;
  a.Bref[idx] = B;   // the new deviations refer to this step's B
  if (a.fxx) eddington_factors(a, idx, E, nxx, nxy, nyy);
}

// One thread per (track, sense, polar chunk, group), groups fastest, tracks longest first (so that the last blocks are
// short ones): NPT polar cosines, a divisor of their number.  The record of step s + 2 and the cell entry and state of step s + 1 are
// loaded before step s is computed.
template <int NPT, int EXTRA>
__global__ void __launch_bounds__(128, NPT >= 4 ? 3 : 4) sweep_fp64_kernel(PlanView v, SweepArgs a, int n_chunks) {
  constexpr bool FACES = EXTRA == kSweepFaces, BAL = EXTRA == kSweepBalance;
  static_assert(!BAL || NPT == 1, "the balance check follows one ray per thread");
  __shared__ u64 table[64];
  chain_next();
  if (threadIdx.x < 64) table[threadIdx.x] = kExp2Table[threadIdx.x];
  __syncthreads();
  const int NP = v.n_polar, Q = v.G * NP;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= v.n_tracks * 2 * v.G * n_chunks) return;
  const int g = (int)(idx % v.G);
  int64_t rest = idx / v.G;
  const int p0 = (int)(rest % n_chunks) * NPT;
  rest /= n_chunks;
  const int sense = (int)(rest & 1);
  const TrackDev tr = v.tracks[v.track_order[rest >> 1]];
  const PairDev pr = v.pairs[tr.pair];
  const PolarFix *pf = v.polar_fix + tr.pair * NP + p0;
  const double cx = sense ? -pr.c : pr.c, cy = sense ? -pr.s : pr.s;
  const double cxx = cx * cx, cxy = cx * cy, cyy = cy * cy;
  double *I = (double *)a.I + (2 * tr.seg_off + (int64_t)sense * tr.nseg) * Q + g * NP + p0;
  const int nseg = tr.nseg;
  const int64_t seg0 = sense ? tr.seg_off + nseg - 1 : tr.seg_off;
  const int sstep = sense ? -1 : 1;
  chain_wait();
  const double Iin = a.bnd[(sense ? tr.entry_minus : tr.entry_plus) * v.G + g];
  const double inv_cdt = a.inv_cdt;
  const bool pairs2 = NPT % 2 == 0;   // 16-byte aligned: even rows, even offset (and the state: launch_sweep_fp64)
  auto load_state = [&](const double *p, double (&d)[NPT]) {
    if (pairs2) {
#pragma unroll
      for (int i = 0; i + 1 < NPT; i += 2) {
        const double2 t = __ldcs(reinterpret_cast<const double2 *>(p + i));
        d[i] = t.x;
        d[i + 1] = t.y;
      }
    } else {
#pragma unroll
      for (int i = 0; i < NPT; ++i) d[i] = __ldcs(p + i);
    }
  };
  auto load_cell = [&](int cell, Cell64 &c) {
    if (a.cell64) {
      // plain loads: the prep kernel writes the table while this kernel may already be resident (chain_wait)
      const double2 *q = reinterpret_cast<const double2 *>(a.cell64 + (int64_t)cell * v.G + g);
      const double2 x = q[0], y = q[1];
      c.kt = x.x;
      c.r = x.y;
      c.B = y.x;
      c.dB = y.y;
    } else {
      const int64_t i = (int64_t)g * v.ncell + cell;
      c = cell64(a.kappa[i], a.B[i], a.Bref[i], inv_cdt);
    }
  };

  double psi[NPT], cur[NPT], nxt[NPT];
#pragma unroll
  for (int p = 0; p < NPT; ++p) psi[p] = cur[p] = nxt[p] = 0.0;
  int cell = 0, cell1 = 0;
  double len = 0.0, af = 0.0, len1 = 0.0, af1 = 0.0;
  Cell64 c{}, c1{};
  if (nseg > 0) {
    cell = v.seg_cell[seg0];
    len = v.seg_len[seg0];
    af = v.seg_afrac[seg0];
    load_cell(cell, c);
    load_state(I, cur);
  }
  if (nseg > 1) {
    cell1 = v.seg_cell[seg0 + sstep];
    len1 = v.seg_len[seg0 + sstep];
    af1 = v.seg_afrac[seg0 + sstep];
  }
  double Bprev = Iin;   // the boundary acts as the cell before the first
  double rb = 0.0, sb = 0.0;   // MOLC_BALANCE: sum of tau (d - psibar) and the magnitudes of the terms
  for (int s = 0; s < nseg; ++s) {
    int cell2 = 0;
    double len2 = 0.0, af2 = 0.0;
    if (s + 1 < nseg) {
      load_cell(cell1, c1);
      load_state(I + Q, nxt);
    }
    if (s + 2 < nseg) {
      const int64_t q = seg0 + (int64_t)(s + 2) * sstep;
      cell2 = v.seg_cell[q];
      len2 = v.seg_len[q];
      af2 = v.seg_afrac[q];
    }
    const double jump = Bprev - c.B;
    const double kl = c.kt * len;
    int ek;
    const u64 Mk = double_mantissa(kl, ek);
    double E1[NPT], f[NPT];
    bool thin[NPT];
    if ((unsigned)(ek + 900) <= 1800u) {   // not so for zeros, negatives, infinities and NaN
      const u64 Mr = fixed_reciprocal(Mk);
#pragma unroll
      for (int p = 0; p < NPT; ++p) attenuation_fixed(Mk, ek, Mr, load_polar(pf + p), table, E1[p], f[p], thin[p]);
    } else {
#pragma unroll
      for (int p = 0; p < NPT; ++p)
        attenuation_fp64(kl * v.polar[tr.pair * NP + p0 + p].inv_sinz, E1[p], f[p], thin[p]);
    }
    double F0 = 0.0, F1 = 0.0, F2 = 0.0, S[3] = {0.0, 0.0, 0.0};
    if constexpr (BAL) sb += fabs(jump);
#pragma unroll
    for (int p = 0; p < NPT; ++p) {
      const double pin = psi[p] + jump;
      if constexpr (FACES) {   // Eq. (16): omega w times the intensity at the segment's upwind face
        const double in = pin + c.B;
        F0 = fma(pf[p].w, in, F0);
        F1 = fma(pf[p].ws, in, F1);
        F2 = fma(pf[p].wss, in, F2);
      }
      const double d = fma(cur[p], c.r, c.dB);
      const double x = pin - d;
      const double pb = fma(x, E1[p], d);
      // thin: psi_in - (psi_in - d)(1 - e^-tau), the change to its own accuracy; thick: d + (psi_in - d) e^-tau,
      // the transmitted part to its own accuracy
      psi[p] = fma(thin[p] ? -x : x, f[p], thin[p] ? pin : d);
      cur[p] = pb;
      S[0] = fma(pf[p].w, pb, S[0]);
      S[1] = fma(pf[p].ws, pb, S[1]);
      S[2] = fma(pf[p].wss, pb, S[2]);
      if constexpr (BAL) {
        const double tau = kl * v.polar[tr.pair * NP + p0 + p].inv_sinz;
        rb += tau * (d - pb);
        sb += fabs(c.B + pin) + fabs(c.B + psi[p]) + fabs(pin) + fabs(psi[p]) +
              tau * (fabs(c.B + d) + fabs(c.B + pb));
      }
    }
    if (pairs2) {
#pragma unroll
      for (int i = 0; i + 1 < NPT; i += 2) __stcs(reinterpret_cast<double2 *>(I + i), make_double2(cur[i], cur[i + 1]));
    } else {
#pragma unroll
      for (int i = 0; i < NPT; ++i)
        __stcs(I + i, cur[i]);
    }
    if constexpr (FACES) {
      const int2 fc = v.seg_face[seg0 + (int64_t)s * sstep];
      double *fa = v.facc + (int64_t)(sense ? fc.y : fc.x) * kOutputs * v.G + g;
      F0 *= tr.width;
      F1 *= tr.width;
      F2 *= tr.width;
      atomicAdd(fa, F0);
      atomicAdd(fa + v.G, F1 * cx);
      atomicAdd(fa + 2 * v.G, F1 * cy);
      atomicAdd(fa + 3 * v.G, F2 * cxx);
      atomicAdd(fa + 4 * v.G, F2 * cxy);
      atomicAdd(fa + 5 * v.G, F2 * cyy);
    }
    double *acc = a.acc + (int64_t)cell * kOutputs * v.G + g;
#pragma unroll
    for (int k = 0; k < 3; ++k) S[k] *= af;
    atomicAdd(acc, S[0]);
    atomicAdd(acc + v.G, S[1] * cx);
    atomicAdd(acc + 2 * v.G, S[1] * cy);
    atomicAdd(acc + 3 * v.G, S[2] * cxx);
    atomicAdd(acc + 4 * v.G, S[2] * cxy);
    atomicAdd(acc + 5 * v.G, S[2] * cyy);
    Bprev = c.B;
    I += Q;
    cell = cell1;
    len = len1;
    af = af1;
    c = c1;
    cell1 = cell2;
    len1 = len2;
    af1 = af2;
#pragma unroll
    for (int p = 0; p < NPT; ++p) cur[p] = nxt[p];
  }
  if constexpr (BAL) {
    if (nseg > 0) ray_balance_max(v.balance, Iin - (psi[0] + Bprev) + rb, sb, 1.0);
  }
}

// Blocks of the preparation; whether an FP64 step is chained.
int prep_blocks_fp64(const PlanView &v) {
  return (int)std::min<int64_t>(((int64_t)v.G * v.ncell + 255) / 256, 152 * 8);
}
bool chained(const PlanView &v) { return few_walks(v) && prep_blocks_fp64(v) <= 48; }

template <int NPT, int EXTRA>
cudaError_t launch_fp64(const PlanView &v, const SweepArgs &a, cudaStream_t st) {
  const int n_chunks = v.n_polar / NPT;
  const int64_t blocks = (v.n_tracks * 2 * (int64_t)v.G * n_chunks + 127) / 128;
  if (blocks > 0x7fffffff) return cudaErrorInvalidConfiguration;
  return launch_chained(chained(v), sweep_fp64_kernel<NPT, EXTRA>, (unsigned)blocks, 128, 0, st, v, a, n_chunks);
}

}  // namespace

cudaError_t launch_prep_fp64(const PlanView &v, const SweepArgs &a, cudaStream_t st) {
  prep_fp64_kernel<<<(unsigned)prep_blocks_fp64(v), 256, 0, st>>>(v, a);
  return cudaGetLastError();
}

cudaError_t launch_finalize_fp64(const PlanView &v, const SweepArgs &a, cudaStream_t st) {
  const dim3 grid((unsigned)((v.ncell + kFinalCells - 1) / kFinalCells),
                  (unsigned)((v.G + kFinalGroups - 1) / kFinalGroups));
  return launch_chained(chained(v), finalize_fp64_kernel, grid, kFinalCells * kFinalGroups, 0, st, v, a);
}

cudaError_t launch_sweep_fp64(const PlanView &v, const SweepArgs &a, cudaStream_t st) {
  if (v.balance) return launch_fp64<1, kSweepBalance>(v, a, st);
  if (v.facc) return launch_fp64<1, kSweepFaces>(v, a, st);
  // Polar cosines one thread carries: the largest divisor of their number, up to 8, that leaves 16 warps an SM
  // (152 x 512 threads).  More of them share a segment's products and atomics, but with fewer threads the short
  // characteristics end early and the long ones run on alone: 17 groups, 8 polar cosines, 128^2 cells (355k walks)
  // 13.1 ms with 1, 9.4 with 2, 8.0 with 4, 7.7 with 8; 7 groups, 3 polar cosines, 75 x 52 cells (23k walks) 250 us
  // with 1 and 317 with 3; 7 groups, 4 polar cosines, 150 x 100 cells (45k walks) 838 us with 1, 743 with 2, 930 with 4.
  constexpr int64_t kEnough = 152 * 512;
  const int64_t walks = v.n_tracks * 2 * (int64_t)v.G;
  int npt = v.n_polar < 8 ? v.n_polar : 8;
  // an even number is loaded in pairs: not from a state that starts 8 bytes past a 16-byte boundary
  const bool pairs = ((uintptr_t)a.I & 15) == 0;
  while (npt > 1 && (v.n_polar % npt || walks * (v.n_polar / npt) < kEnough || (npt % 2 == 0 && !pairs))) --npt;
  switch (npt) {
    case 8: return launch_fp64<8, kSweepPlain>(v, a, st);
    case 7: return launch_fp64<7, kSweepPlain>(v, a, st);
    case 6: return launch_fp64<6, kSweepPlain>(v, a, st);
    case 5: return launch_fp64<5, kSweepPlain>(v, a, st);
    case 4: return launch_fp64<4, kSweepPlain>(v, a, st);
    case 3: return launch_fp64<3, kSweepPlain>(v, a, st);
    case 2: return launch_fp64<2, kSweepPlain>(v, a, st);
    default: return launch_fp64<1, kSweepPlain>(v, a, st);
  }
}

}  // namespace molc
