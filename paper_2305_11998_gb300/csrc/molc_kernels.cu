// CUDA kernels of libmolc (sm_103a): the MOLC high-order sweep of Sec. 3 in two precisions, the cell
// assembly of the moments, the Eddington closure and the intensity-state utilities.
//
// Both sweeps walk each characteristic in the deviation form psi = I - B_i (B_i the Planck intensity of
// the current cell).  With S = Q / kappa~ (Eq. 11) and E1(tau) = (1 - e^-tau) / tau, Eqs. (12)-(13) become
//     psi_out  = d + (psi_in - d) e^-tau,     psibar = d + (psi_in - d) E1(tau),
//     d = S - B_i = (I^{n-1} - B_i) / (c dt kappa~),
// (alpha I_s + (1 - alpha) I_{s+1} = S + (I_s - S) E1 exactly), and at a cell crossing
// psi_in(next) = psi_out + (B_prev - B_next).  The stored state is the deviation delta = Ibar - B_ref of each
// segment average from the Planck intensity B_ref its cell had when it was written, so
// d = (delta + B_ref - B) / (c dt kappa~) keeps the precision of the deviation (exactly 0 after
// molc_intensity_init, in any precision).  The cell moments then carry the deviations, and the B_i part
// is added analytically from per-cell geometric moments (it cancels exactly in F: the two senses of a track
// have opposite Omega and equal areas).  This keeps the cancelling sums F and N_xy accurate in optically
// thick cells, where |F| can be ~1e-8 c E.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "molc_device.cuh"
#include "molc_internal.h"

namespace molc {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// Track holding row r of the intensity layout (rows are (track, sense, step); a track owns 2 nseg rows).
__device__ __forceinline__ int64_t find_track(const TrackDev *tr, int64_t T, int64_t row) {
  int64_t lo = 0, hi = T - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (2 * tr[mid].seg_off <= row)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// ---------------------------------------------------------------------------------------------------------
// prep (FP32): input checks, and per (chunk, cell, group) {kappa~, 1/(c dt kappa~), B_hi, B_lo}
// with B = B_hi + B_lo split so that B differences between neighbouring cells keep ~48 bits.
// ---------------------------------------------------------------------------------------------------------
constexpr int kPrepCells = 32;   // cells per tile of prep_kernel

// Tiles of kPrepCells cells x the groups of one chunk: [g][cell] inputs are read along cells, the
// [chunk][cell][gc] tables are staged in shared memory and written out contiguously.  A block takes tiles
// tile0, tile0 + tstride, ...; check_bnd: this block also checks the boundary values.
__device__ __forceinline__ void prep_tiles(const PlanView &v, const SweepArgs &a, const Layout &L,
                                           int chunk, int tile0, int tstride, bool check_bnd) {
  __shared__ float4 t4[kPrepCells * 32];
  __shared__ float t1[kPrepCells * 32];
  const float inv_cdt_f = (float)a.inv_cdt;
  const double sc = a.scale[0];
  const int g0 = chunk * L.gc;
  const int gcount = min(L.gc, v.G - g0);
  bool bad = false, range = false;
  const int n_tiles = (v.ncell + kPrepCells - 1) / kPrepCells;
  for (int tile = tile0; tile < n_tiles; tile += tstride) {
    const int c0 = tile * kPrepCells;
    const int nc = min(kPrepCells, v.ncell - c0);
#pragma unroll 4
    for (int k = threadIdx.x; k < kPrepCells * gcount; k += blockDim.x) {
      const int gl = k / kPrepCells, c = k - gl * kPrepCells;
      if (c >= nc) continue;
      const int64_t idx = (int64_t)(g0 + gl) * v.ncell + c0 + c;
      const double kap = a.kappa[idx], B = a.B[idx];
      bad |= bad_input(kap) | bad_input(B);
      // FP64 only where a difference or a split needs it (the FP64 pipe is narrow): kappa~ and
      // 1/(c dt kappa~) are rounded to FP32 anyway and are formed in FP32
      const float kt = (float)(kap + a.inv_cdt);
      const float r = __fdiv_rn(inv_cdt_f, kt);
      const double Bs = B * sc;
      // !(Bs < kScaledMax) on the bits: signed order is value order for non-negative doubles and -0
      range |= __double_as_longlong(Bs) >= __double_as_longlong(kScaledMax);
      const float bhi = (float)Bs;
      const float blo = (float)(Bs - f32_to_f64_exact(bhi));
      t4[c * gcount + gl] = make_float4(kt, r, bhi, blo);
      t1[c * gcount + gl] = (float)((a.Bref[idx] - B) * sc) * r;
    }
    __syncthreads();
    // [chunk][cell][gc]: the chunk's stride is gc also in a partial last chunk (as the sweep reads it)
    const int64_t o = (int64_t)g0 * v.ncell + (int64_t)c0 * L.gc;
    for (int k = threadIdx.x; k < nc * gcount; k += blockDim.x) {
      const int c = k / gcount, gl = k - c * gcount;
      a.cdat[o + (int64_t)c * L.gc + gl] = t4[k];
      a.cdB[o + (int64_t)c * L.gc + gl] = t1[k];
    }
    __syncthreads();
  }
  if (check_bnd)
    for (int i = threadIdx.x; i < 4 * v.G; i += blockDim.x) {
      bad |= bad_input(a.bnd[i]);
      range |= !(a.bnd[i] * sc < kScaledMax);
    }
  if (bad) atomicOr(v.status, kStatusNonfinite);
  if (range && !bad) atomicOr(v.status, kStatusRange);
}

__global__ void __launch_bounds__(128) prep_kernel(PlanView v, SweepArgs a, Layout L) {
  chain_next();
  chain_wait();
  prep_tiles(v, a, L, blockIdx.y, blockIdx.x, gridDim.x, blockIdx.x == 0 && blockIdx.y == 0);
}

// Batched (FP32): block j prepares tile map[j].z of chunk map[j].y of instance map[j].x.
__global__ void __launch_bounds__(128) prep_batch_kernel(const BatchInst *inst, const int4 *map) {
  const int4 m = map[blockIdx.x];
  const BatchInst &b = inst[m.x];
  prep_tiles(b.v, b.a, b.L, m.y, m.z, 1 << 30, m.w != 0);
}

// ---------------------------------------------------------------------------------------------------------
// FP32 production sweep.  One thread per (track, sense, group): the thread walks its track in its sense and
// carries all NP polar cosines of the azimuth in registers (the in-plane track is shared by them).  Threads of
// a warp hold consecutive groups of the same track-sense, so the record and cell-table loads are shared and
// coalesced; the previous-step deviations stream in and out in the bundle layout (a block's 128 threads read
// and write 128 * NP contiguous values per step).  The sweep does no reduction: the cell moments are gathered
// afterwards from the swept state (moments_fp32_kernel).
// ---------------------------------------------------------------------------------------------------------

// 2^x (ex2.approx.ftz.f32: the SFU's base-2 exponential).
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// E1 = (1 - e^-tau)/tau, e^-tau and, for tau < 1/2, om = 1 - e^-tau in FP32, from a = tau/2.  With
// h = e^-a = 2^(-a log2 e):
//   tau < 1/2:  E1 = h sinh(a) / a, the even Taylor series in y = a^2 to y^3 (truncation < 5e-11 relative),
//               free of cancellation, and om = tau E1 (= 2 h sinh(a));
//   tau >= 1/2: E1 = (1 - e^-tau) / tau (1 - e^-tau > 0.39, no cancellation).
// e^-tau = h^2.  inv_tau is 1/tau.  The outgoing intensity is taken as psi_in - (psi_in - d) om below tau = 1/2
// and as d + (psi_in - d) e^-tau above: equal in exact arithmetic, but across a thin segment the first keeps the
// change to the relative accuracy of om where the second would carry the rounding of e^-tau on all of psi_in - d,
// and across a thick one the second keeps the small transmitted part to the relative accuracy of e^-tau.
__device__ __forceinline__ void attenuation(float a, float inv_tau, float &E1, float &om, float &ex, bool &thin) {
  constexpr float kMinusLog2e = -1.4426950408889634f;
  const float h = ex2_approx(a * kMinusLog2e);
  ex = h * h;
  const float y = a * a;
  float p = fmaf(y, 1.f / 5040.f, 1.f / 120.f);
  p = fmaf(p, y, 1.f / 6.f);
  p = fmaf(p, y, 1.f);
  const float hp = h * p;
  thin = a < 0.25f;
  E1 = thin ? hp : (1.f - ex) * inv_tau;
  om = (a + a) * hp;
}

// L2 eviction policy (sm_80+ createpolicy) for the streamed state, which each pass touches once: evict-first,
// so that the cell tables and segment records stay in L2.
__device__ __forceinline__ unsigned long long policy_evict_first() {
  unsigned long long p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// NP consecutive FP32 deviations of one thread: vector accesses where the alignment allows (the row offset is
// a multiple of NP elements and the state is 256-byte aligned), evict-first in L2, no L1 allocation.
template <int NP>
__device__ __forceinline__ void load_dev(const float *p, float (&v)[NP], unsigned long long pol) {
  if constexpr (NP % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 4)
      asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
          : "=f"(v[i]), "=f"(v[i + 1]), "=f"(v[i + 2]), "=f"(v[i + 3])
          : "l"(p + i), "l"(pol));
  } else if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 2)
      asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;"
          : "=f"(v[i]), "=f"(v[i + 1])
          : "l"(p + i), "l"(pol));
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i)
      asm volatile("ld.global.L1::no_allocate.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v[i]) : "l"(p + i), "l"(pol));
  }
}
// The same through L2 with the default policy (ld.global.cg): the moment gather reads pieces of the state that
// share sectors with pieces other cells read at about the same time.
template <int NP>
__device__ __forceinline__ void load_dev_cg(const float *p, float (&v)[NP]) {
  if constexpr (NP % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 4) {
      const float4 t = __ldcg(reinterpret_cast<const float4 *>(p + i));
      v[i] = t.x;
      v[i + 1] = t.y;
      v[i + 2] = t.z;
      v[i + 3] = t.w;
    }
  } else if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 2) {
      const float2 t = __ldcg(reinterpret_cast<const float2 *>(p + i));
      v[i] = t.x;
      v[i + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) v[i] = __ldcg(p + i);
  }
}
template <int NP>
__device__ __forceinline__ void store_dev(float *p, const float (&v)[NP], unsigned long long pol) {
  if constexpr (NP % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 4)
      asm volatile("st.global.L1::no_allocate.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p + i),
                   "f"(v[i]), "f"(v[i + 1]), "f"(v[i + 2]), "f"(v[i + 3]), "l"(pol)
                   : "memory");
  } else if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 2)
      asm volatile("st.global.L1::no_allocate.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p + i), "f"(v[i]),
                   "f"(v[i + 1]), "l"(pol)
                   : "memory");
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i)
      asm volatile("st.global.L1::no_allocate.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(p + i), "f"(v[i]), "l"(pol)
                   : "memory");
  }
}

// One cp.async of `bytes` (4, 8 or 16) from global to shared memory; with the L2 policy `pol` when HINT.  The
// hinted form is used only where every copy's address is formed in registers with no constant offset folded into
// the instruction (up to 4 polar cosines: one copy per thread or one piece per lane); the other polar counts copy
// several pieces at constant offsets from one address and take the plain form.
template <bool HINT, int BYTES>
__device__ __forceinline__ void cp_async_piece(unsigned dst, const float *src, unsigned long long pol) {
  static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async copies 4, 8 or 16 bytes");
  if constexpr (HINT) {
    if constexpr (BYTES == 16)
      asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(pol)
                   : "memory");
    else
      asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], %2, %3;" ::"r"(dst), "l"(src),
                   "n"(BYTES), "l"(pol)
                   : "memory");
  } else {
    if constexpr (BYTES == 16)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
  }
}

// Asynchronous copies (cp.async, sm_80+) of NP consecutive FP32 deviations from global to shared memory:
// 16-byte pieces where NP * 4 bytes allow, else 8- or 4-byte pieces (the thread's deviations start at a multiple
// of NP * 4 bytes of a 256-byte aligned state).  The streamed state is read with the L2 policy `pol`
// (evict-first), so that it does not push the cell tables and segment records out of L2 (up to 4 polar cosines).
template <int NP>
__device__ __forceinline__ void copy_dev_async(float *dst_smem, const float *src, unsigned long long pol) {
  constexpr bool kHint = NP <= 4;
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
  if constexpr (NP % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 4) cp_async_piece<kHint, 16>(d + 4 * i, src + i, pol);
  } else if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 2) cp_async_piece<kHint, 8>(d + 4 * i, src + i, pol);
  } else {
#pragma unroll
    for (int i = 0; i < NP; ++i) cp_async_piece<kHint, 4>(d + 4 * i, src + i, pol);
  }
}
// Warp-cooperative forms for odd NP: the 32 threads of a warp hold 32 x NP consecutive floats of a bundle step
// slot (128 NP bytes, 16-byte aligned), moved as 8 NP pieces of 16 bytes by the first 8 NP lanes (one
// instruction per lane for NP <= 4) instead of NP scalar accesses per thread.
template <int NP>
__device__ __forceinline__ void copy_warp_chunk_async(float *dst_smem, const float *src, int lane,
                                                      unsigned long long pol) {
  constexpr int kPieces = 8 * NP;
  constexpr bool kHint = NP <= 4;
#pragma unroll
  for (int j = 0; j < (kPieces + 31) / 32; ++j) {
    const int k = lane + 32 * j;
    if (k < kPieces)
      cp_async_piece<kHint, 16>((unsigned)__cvta_generic_to_shared(dst_smem + 4 * k), src + 4 * k, pol);
  }
}
template <int NP>
__device__ __forceinline__ void store_warp_chunk(float *dst, const float *src_smem, int lane,
                                                 unsigned long long pol) {
  constexpr int kPieces = 8 * NP;
#pragma unroll
  for (int j = 0; j < (kPieces + 31) / 32; ++j) {
    const int k = lane + 32 * j;
    if (k < kPieces) {
      const float4 t = *reinterpret_cast<const float4 *>(src_smem + 4 * k);
      asm volatile("st.global.L1::no_allocate.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(dst + 4 * k),
                   "f"(t.x), "f"(t.y), "f"(t.z), "f"(t.w), "l"(pol)
                   : "memory");
    }
  }
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void copy16_async(void *dst_smem, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst_smem)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy4_async(void *dst_smem, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst_smem)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ int2 ld_record(const int2 *p) {
  int2 v;
  // volatile: a load the compiler cannot see as one must not be executed speculatively (callers guard the
  // address range with a condition)
  asm volatile("ld.global.nc.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}

// Software pipeline of the FP32 sweep, per thread, in rings of D slots (D = staging depth, chosen per plan by
// the autotuner; the step loop is unrolled by D so that every slot index is a constant): at step s the thread
//   - issues asynchronous copies of its previous-step deviations for step s+D-1 and of the cell table entry of
//     step s+D-2 (whose record arrived two steps earlier) into shared memory, as one cp.async group,
//   - waits until the groups holding step s's deviations and table entry have landed,
//   - computes step s and stores its new deviations to global memory,
//   - loads the record of step s+D into a register.
// Group accounting: the prologue commits D-1 groups (deviations of steps 0..D-2, table entries of steps
// 0..D-3) and step s commits one; step s's deviations are in group s and its table entry in group s+1 (group s
// for s <= D-3), so waiting until at most D-2 groups are pending is enough.
// For odd NP the deviations of a step are copied for the whole warp by its first 8 NP lanes (every lane then
// runs the warp's longest track's steps, the copies and commits warp-uniform, a __syncwarp making the landed
// copies visible to the other lanes and ordering the reads of a slot before its refill), and the new deviations
// go back through the slot: each thread writes its own, the warp stores the slot's chunk in 16-byte pieces.  A thread whose track has ended leaves its part of the slot as it was copied,
// so the padding it stores back is unchanged.
// Shared memory of one FP32 sweep block: D staged steps of its 128 threads' deviations, cell-table entries and
// B_ref differences.
template <int NP, int D>
struct __align__(16) SweepSmem {
  float dev[D][kSweepBlock * NP];
  float4 tab[D][kSweepBlock];
  float dB[D][kSweepBlock];
};

template <int NP, int D, int EXTRA = kSweepPlain>
__device__ __forceinline__ void sweep_fp32_body(const PlanView &v, const SweepArgs &a, const Layout &L, int bundle,
                                                SweepSmem<NP, D> &sm) {
  static_assert(D >= 3, "the staging depth needs D >= 3");
  constexpr bool FACES = EXTRA == kSweepFaces, BAL = EXTRA == kSweepBalance;
  constexpr bool COOP = NP % 2 != 0;       // warp-cooperative copies and stores of the deviations (odd NP; even NP
  constexpr bool COOP_ST = COOP;           // already copies 8 or 16 bytes per thread, and NP = 2 measured slower)
  constexpr int kSteps = D;
  auto &sdev = sm.dev;
  auto &stab = sm.tab;
  auto &sdB = sm.dB;
  const int tid = threadIdx.x;
  const int64_t item = (int64_t)bundle * kSweepBlock + tid;
  const bool live = item < a.n_items;
  const int2 it = live ? a.items[item] : make_int2(0, 0);
  const TrackDev tr = v.tracks[it.x];
  const int sense = it.y & 1, gi = (it.y >> 1) & 0x7fff, ch = it.y >> 16;
  const int g0 = ch * L.gc;
  const int gcount = min(L.gc, v.G - g0);
  const int g = g0 + gi;
  const int nseg = live ? tr.nseg : 0;
  // warp-uniform trip count
  int nmax = nseg;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nmax = max(nmax, __shfl_xor_sync(kFull, nmax, o));
  if (nmax == 0) return;

  const unsigned long long pol_stream = policy_evict_first();
  // floats between consecutive steps of one item (bundle layout); a run-time value, so that the copies below
  // address through registers
  const int64_t stride = (int64_t)kSweepBlock * v.n_polar;
  float *I = (float *)a.I + (v.boff[bundle] * kSweepBlock + tid) * NP;
  const int lane = tid & 31, wofs = (tid & ~31) * NP;   // this warp's chunk in a slot (COOP)
  float *Iw = (float *)a.I + v.boff[bundle] * kSweepBlock * NP + wofs;
  const int nlim = COOP ? nmax : nseg;   // steps this thread copies and commits for
  const int2 *rec = v.seg32 + (sense ? tr.seg_off + nseg - 1 : tr.seg_off);
  const int rstep = sense ? -1 : 1;
  const int64_t cbase = (int64_t)ch * v.ncell * L.gc + gi;
  const float4 *cd = a.cdat + cbase;
  const float *cdB = a.cdB + cbase;

  float half_inv_sinz[NP], sinz[NP], wf[FACES ? NP : 1];   // 1/(2 sin zeta): tau/2 = kappa~ l half_inv_sinz
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const PolarDev pd = v.polar[tr.pair * NP + p];
    half_inv_sinz[p] = 0.5f * pd.inv_sinzf;
    sinz[p] = pd.sinzf;
    if constexpr (FACES) wf[p] = pd.wf;
  }
  // face moments (Eq. 16): faces of this sense's segments, in traversal order like the records
  const int2 *sface = FACES ? v.seg_face + (sense ? tr.seg_off + nseg - 1 : tr.seg_off) : nullptr;
  const float fx = FACES ? (float)((sense ? -1.0 : 1.0) * v.pairs[tr.pair].c) : 0.f;
  const float fy = FACES ? (float)((sense ? -1.0 : 1.0) * v.pairs[tr.pair].s) : 0.f;
  const float width = FACES ? (float)tr.width : 0.f;
  // records of steps 0..D-1; then everything the kernels before this one write
  int2 recs[kSteps];
#pragma unroll
  for (int k = 0; k < kSteps; ++k) recs[k] = k < nseg ? ld_record(rec + k * rstep) : make_int2(0, 0);
  chain_wait();
  // entering intensity (scaled), split like B so that I_in - B keeps the precision of the difference
  const double bin = live ? a.bnd[(sense ? tr.entry_minus : tr.entry_plus) * v.G + g] * a.scale[0] : 0.0;
  const float in_hi = (float)bin, in_lo = (float)(bin - (double)in_hi);
  const float rescale = (float)a.scale[3];   // power of two: the stored deviations to this step's scale

  // prologue: groups 0..D-2 = {deviations k, table k (k <= D-3)}
#pragma unroll
  for (int k = 0; k < kSteps - 1; ++k) {
    if constexpr (COOP) {
      if (k < nmax) copy_warp_chunk_async<NP>(&sdev[k][wofs], Iw + k * stride, lane, pol_stream);
    }
    if (k < nseg) {
      if constexpr (!COOP) copy_dev_async<NP>(&sdev[k][tid * NP], I + k * stride, pol_stream);
      if (k < kSteps - 2) {
        copy16_async(&stab[k][tid], cd + (int64_t)recs[k].x * L.gc);
        copy4_async(&sdB[k][tid], cdB + (int64_t)recs[k].x * L.gc);
      }
    }
    cp_async_commit();
  }
  float psi[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) psi[p] = 0.f;
  float bhi_prev = in_hi, blo_prev = in_lo;   // the boundary acts as the "previous cell" of step 0
  // MOLC_BALANCE, in FP64 from this sweep's FP32 values: per polar cosine the sum of tau (d - psibar) and of the
  // magnitudes of the terms; the crossing steps are common to the polar cosines; B of the last cell
  double rb[BAL ? NP : 1], sb[BAL ? NP : 1], jsum = 0.0, blast = 0.0;
  if constexpr (BAL) {
#pragma unroll
    for (int p = 0; p < NP; ++p) rb[p] = sb[p] = 0.0;
  }
  for (int s0 = 0; s0 < nmax; s0 += kSteps) {
#pragma unroll
    for (int u = 0; u < kSteps; ++u) {
      const int s = s0 + u;
      if (s < nlim) {
        // group s+D-1: deviations of step s+D-1, table entry of step s+D-2
        if constexpr (COOP) {
          __syncwarp();   // every lane is done with the slot refilled here (read at step s-1)
          if (s + kSteps - 1 < nmax)
            copy_warp_chunk_async<NP>(&sdev[(u + kSteps - 1) % kSteps][wofs], Iw + (kSteps - 1) * stride, lane,
                                      pol_stream);
        } else {
          if (s + kSteps - 1 < nseg)
            copy_dev_async<NP>(&sdev[(u + kSteps - 1) % kSteps][tid * NP], I + (kSteps - 1) * stride, pol_stream);
        }
        if (s + kSteps - 2 < nseg) {
          const int c2 = recs[(u + kSteps - 2) % kSteps].x;
          copy16_async(&stab[(u + kSteps - 2) % kSteps][tid], cd + (int64_t)c2 * L.gc);
          copy4_async(&sdB[(u + kSteps - 2) % kSteps][tid], cdB + (int64_t)c2 * L.gc);
        }
        cp_async_commit();
        cp_async_wait<kSteps - 2>();   // deviations and table entry of step s have landed
        if constexpr (COOP) __syncwarp();   // ... including the pieces other lanes copied
        if (s < nseg) {
          float dv[NP];
          if constexpr (NP % 4 == 0) {
#pragma unroll
            for (int p = 0; p < NP; p += 4) {
              const float4 t4 = *reinterpret_cast<const float4 *>(&sdev[u][tid * NP + p]);
              dv[p] = t4.x;
              dv[p + 1] = t4.y;
              dv[p + 2] = t4.z;
              dv[p + 3] = t4.w;
            }
          } else {
#pragma unroll
            for (int p = 0; p < NP; ++p) dv[p] = sdev[u][tid * NP + p];
          }
          const float4 q = stab[u][tid];
          const float qy = q.y * rescale;   // rescale (a power of two) brings the stored deviations to this scale
          const float dB = sdB[u][tid];
          // step s
          const float len = __int_as_float(recs[u].y);
          const float jump = (bhi_prev - q.z) + (blo_prev - q.w);
          const float kl = q.x * len;
          const float rkl = rcp_approx(kl);
#pragma unroll
          for (int p = 0; p < NP; ++p) psi[p] += jump;
          double bcell = 0.0;
          if constexpr (BAL) {
            jsum += fabs(f32_to_f64_exact(jump));
            bcell = f32_to_f64_exact(q.z) + f32_to_f64_exact(q.w);
            blast = bcell;
          }
          if constexpr (FACES) {
            // the intensity entering the segment, in scaled units: psi (relative to this cell) + B of this cell
            const float Bc = q.z + q.w;
            float S0 = 0.f, S1 = 0.f, S2 = 0.f;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
              const float t0 = wf[p] * (psi[p] + Bc);
              S0 += t0;
              const float t1 = t0 * sinz[p];
              S1 += t1;
              S2 = fmaf(t1, sinz[p], S2);
            }
            const int2 fc = __ldg(sface + s * rstep);
            double *fa = v.facc + ((int64_t)ch * v.n_faces + (sense ? fc.y : fc.x)) * kOutputs * L.gc + gi;
            S0 *= width;
            S1 *= width;
            S2 *= width;
            atomicAdd(fa, f32_to_f64(S0));
            atomicAdd(fa + L.gc, f32_to_f64(fx * S1));
            atomicAdd(fa + 2 * L.gc, f32_to_f64(fy * S1));
            atomicAdd(fa + 3 * L.gc, f32_to_f64(fx * fx * S2));
            atomicAdd(fa + 4 * L.gc, f32_to_f64(fx * fy * S2));
            atomicAdd(fa + 5 * L.gc, f32_to_f64(fy * fy * S2));
          }
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            float E1, om, ex;
            bool thin;
            const float ahalf = kl * half_inv_sinz[p];   // tau / 2
            attenuation(ahalf, sinz[p] * rkl, E1, om, ex, thin);
            const float d = fmaf(dv[p], qy, dB);
            const float pin = psi[p];
            const float x = pin - d;
            dv[p] = fmaf(x, E1, d);
            psi[p] = thin ? fmaf(-x, om, pin) : fmaf(x, ex, d);
            if constexpr (BAL) {
              const double tau = 2.0 * f32_to_f64_exact(ahalf), dd = f32_to_f64_exact(d),
                           pb = f32_to_f64_exact(dv[p]);
              rb[p] += tau * (dd - pb);
              const double pi = f32_to_f64_exact(pin), po = f32_to_f64_exact(psi[p]);
              sb[p] += fabs(bcell + pi) + fabs(bcell + po) + fabs(pi) + fabs(po) +
                       tau * (fabs(bcell + dd) + fabs(bcell + pb));
            }
        }
        if constexpr (COOP_ST) {
#pragma unroll
          for (int p = 0; p < NP; ++p) sdev[u][tid * NP + p] = dv[p];
        } else {
          store_dev<NP>(I, dv, pol_stream);
        }
        bhi_prev = q.z;
        blo_prev = q.w;
        I += stride;
        if (s + kSteps < nseg) recs[u] = ld_record(rec + (s + kSteps) * rstep);
        }
        if constexpr (COOP_ST) {
          __syncwarp();
          store_warp_chunk<NP>(Iw, &sdev[u][wofs], lane, pol_stream);
        }
        Iw += stride;
      }
    }
  }
  cp_async_wait<0>();
  if constexpr (BAL) {
    if (nseg > 0) {
      const double Iin = f32_to_f64_exact(in_hi) + f32_to_f64_exact(in_lo);
      double R = 0.0, S = 0.0, worst = -1.0;
#pragma unroll
      for (int p = 0; p < NP; ++p) {   // the polar cosine with the largest relative residual
        const double Iout = f32_to_f64_exact(psi[p]) + blast;
        const double r = Iin - Iout + rb[p], sm = sb[p] + jsum;
        const double rel = sm > 0.0 ? fabs(r) / sm : 0.0;
        if (rel > worst) {
          worst = rel;
          R = r;
          S = sm;
        }
      }
      ray_balance_max(v.balance, R, S, a.scale[0]);   // R, S in the state's scaled units
    }
  }
}

// With faces, 6 polar cosines: up to the 128 registers that 4 blocks an SM leave.  Left to itself the compiler takes 96, for a
// fifth block, and the sweep 303 us for 239 (72 x 79 cells, 8 groups, 6 x 32 directions, h/8).
template <int NP, int D, int EXTRA = kSweepPlain>
__global__ void __launch_bounds__(kSweepBlock, EXTRA == kSweepFaces && NP == 6 ? 4 : 0) sweep_fp32_kernel(PlanView v, SweepArgs a, Layout L) {
  __shared__ SweepSmem<NP, D> sm;
  chain_next();
  sweep_fp32_body<NP, D, EXTRA>(v, a, L, v.block_order[blockIdx.x], sm);
}

// Batched: block j sweeps bundle map[j].y of instance map[j].x (blocks of all instances, longest first).
template <int NP, int D>
__global__ void __launch_bounds__(kSweepBlock) sweep_fp32_batch_kernel(const BatchInst *inst, const int2 *map) {
  __shared__ SweepSmem<NP, D> sm;
  const int2 m = map[blockIdx.x];
  const BatchInst &b = inst[m.x];
  sweep_fp32_body<NP, D>(b.v, b.a, b.L, m.y, sm);
}

// FP32 path, cell moments, in two phases.  A cell's (track, sense) segments come as runs of up to kRunSegments track
// segments of one azimuth pair.  First each (run, group) is summed by a thread, in FP32: over the run's segments and
// their two senses, the polar folds S0 = sum_p w_p dev_p, S1 = sum_p w_p sin(zeta_p) dev_p, S2 = sum_p w_p
// sin^2(zeta_p) dev_p of the swept deviations times A/V (S1 signed by the sense).  Then each (cell, group) adds its
// runs' three sums, times (1, Omega, Omega Omega), as unevaluated pairs of FP32 words (hi + lo, TwoSum: a 48-bit
// significand), assembled in FP64:
//   E = (B geo0 + D)/c, F = D_F, N_ab = B geo_ab + D_ab, and B_ref := B.
// Memory latency bounds it: the pieces of a cell (the groups of one segment and sense, contiguous in the state) lie all
// over the state.  With one thread walking a (cell, group)'s list, four pieces at a time, a step's loads waited for that
// step's list words; the lanes of a warp, 2-3 cells, added their pairs' sums at different steps, so that a warp issued
// 146 instructions per segment; and 64^2 cells x 17 groups left half the SMs' slots empty.  So a run's loads, up to eight
// a thread, depend on nothing but words already in shared memory, the runs of a cell are spread over the block, and the
// second phase adds in step.  The FP32 sums run over the same terms in the same order as one thread's walk (run by run,
// segment by segment, + sense before - sense), so the moments do not depend on how cells and runs are shared out.
// A step with one thread walking a cell's list, then so (the gather alone is what changed): 512^2 x 17 groups, 4 polar
// cosines, h/2 3523 -> 3430 us; 128^2 x 17, 8 polar cosines x 64, h/8 3035 -> 2812; 64^2 x 17, 4, h/4 154 -> 137; 40^2 paper
// layout at 1e-3 cm 2191 -> 2081; 16^2 x 4 groups 34.5 -> 28; a batch of 16 problems of 32^2 to 256^2 3709 -> 3520.
__device__ __forceinline__ void two_sum_add(float &hi, float &lo, float x) {
  const float s = __fadd_rn(hi, x);
  const float bp = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(x, bp));
  hi = s;
  lo = __fadd_rn(lo, e);
}

// Tiled sweep: an FP32 partial sum takes at most kPairRun entries (one azimuth pair) before it is added to the two-word sums:
// a cell crossed by many characteristics of one pair (fine ray spacing) keeps the FP32 error of a few terms.
constexpr int kPairRun = 8;

// Assembly of one (cell, group) from its six deviation sums D (state units; is = 1/scale):
//   E = (B geo0 + D0 is)/c, F = D_F is, N_ab = B geo_ab + D_ab is, and B_ref := B.
__device__ __forceinline__ void assemble_cell(const PlanView &v, const SweepArgs &a, int cell, int g,
                                              const double (&D)[kOutputs]) {
  const double is = a.scale[1];   // the deviations are in the state's scaled units (exact power of two)
  const int64_t idx = (int64_t)g * v.ncell + cell;
  const double B = a.B[idx];
  const double E = (B * v.geo[cell] + D[0] * is) * a.inv_c;
  const double nxx = B * v.geo[v.ncell + cell] + D[3] * is;
  const double nxy = B * v.geo[2 * (int64_t)v.ncell + cell] + D[4] * is;
  const double nyy = B * v.geo[3 * (int64_t)v.ncell + cell] + D[5] * is;
  a.out.E[idx] = E;
  a.out.Fx[idx] = D[1] * is;
  a.out.Fy[idx] = D[2] * is;
  a.out.Nxx[idx] = nxx;
  a.out.Nxy[idx] = nxy;
  a.out.Nyy[idx] = nyy;
  a.Bref[idx] = B;   // the new deviations refer to this step's B
  if (a.fxx) eddington_factors(a, idx, E, nxx, nxy, nyy);
}

// Two FP32 values side by side: one instruction rounds both (sm_100+).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 x) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {   // a - b, rounded once
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(b), "l"(pack2(-1.f, -1.f)), "l"(a));
  return r;
}
__device__ __forceinline__ void two_sum_add2(f32x2 &hi, f32x2 &lo, f32x2 x) {   // two_sum_add on each half
  const f32x2 s = add2(hi, x);
  const f32x2 bp = sub2(s, hi);
  const f32x2 e = add2(sub2(hi, sub2(s, bp)), sub2(x, bp));
  hi = s;
  lo = add2(lo, e);
}

// load_dev_cg where `on`, else zeros.
template <int NP>
__device__ __forceinline__ void load_dev_if(bool on, const float *p, float (&v)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) v[i] = 0.f;
  if constexpr (NP % 4 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 4)
      asm("{.reg .pred q;\n setp.ne.s32 q, %5, 0;\n @q ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];}"
          : "+f"(v[i]), "+f"(v[i + 1]), "+f"(v[i + 2]), "+f"(v[i + 3])
          : "l"(p + i), "r"((int)on) : "memory");
  } else if constexpr (NP % 2 == 0) {
#pragma unroll
    for (int i = 0; i < NP; i += 2)
      asm("{.reg .pred q;\n setp.ne.s32 q, %3, 0;\n @q ld.global.cg.v2.f32 {%0, %1}, [%2];}"
          : "+f"(v[i]), "+f"(v[i + 1])
          : "l"(p + i), "r"((int)on) : "memory");
  } else if constexpr (NP >= 5) {
    // an odd number of values starts on an 8-byte boundary or 4 bytes past one: loads of two, and one of the value left
    // over in front or behind
    const bool past = ((uintptr_t)p & 4) != 0;
    float w[NP], one = 0.f;
#pragma unroll
    for (int i = 0; i + 1 < NP; i += 2) {
      w[i] = w[i + 1] = 0.f;
      asm("{.reg .pred q;\n setp.ne.s32 q, %3, 0;\n @q ld.global.cg.v2.f32 {%0, %1}, [%2];}"
          : "+f"(w[i]), "+f"(w[i + 1])
          : "l"(p + i + past), "r"((int)on) : "memory");
    }
    asm("{.reg .pred q;\n setp.ne.s32 q, %2, 0;\n @q ld.global.cg.f32 %0, [%1];}"
        : "+f"(one)
        : "l"(p + (past ? 0 : NP - 1)), "r"((int)on) : "memory");
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const float before = i == 0 ? one : w[i - 1], here = i == NP - 1 ? one : w[i];
      v[i] = past ? before : here;
    }
  } else {   // 1 or 3
#pragma unroll
    for (int i = 0; i < NP; ++i)
      asm("{.reg .pred q;\n setp.ne.s32 q, %2, 0;\n @q ld.global.cg.f32 %0, [%1];}"
          : "+f"(v[i])
          : "l"(p + i), "r"((int)on) : "memory");
  }
}

// N consecutive coefficients, vector loads where a row is padded for them.
template <int NP>
__device__ __forceinline__ void load_fold(const float *p, float (&c)[NP]) {
  if constexpr (NP <= 2) {
#pragma unroll
    for (int i = 0; i < NP; ++i) c[i] = __ldg(p + i);
  } else {
#pragma unroll
    for (int i = 0; i < NP; i += 4) {
      const float4 t = __ldg(reinterpret_cast<const float4 *>(p + i));
      c[i] = t.x;
      if (i + 1 < NP) c[i + 1] = t.y;
      if (i + 2 < NP) c[i + 2] = t.z;
      if (i + 3 < NP) c[i + 3] = t.w;
    }
  }
}

// One block: `units` units of chunk ch.  A unit is a cell, assembled here, or one part of a split cell, whose sums
// go to the scratch partials, summed in order by moments_combine.
template <int NP>
__device__ __forceinline__ void moments_fp32_body(const PlanView &v, const SweepArgs &a, const Layout &L, int ch,
                                                  int64_t block, int units) {
  extern __shared__ __align__(16) unsigned char msmem[];
  chain_next();
  constexpr int kStride = fold_stride(NP), kRow = fold_row(NP);
  constexpr int kTogether = moment_together(NP);   // segments in flight together
  const int g0 = ch * L.gc;
  const int gcount = min(L.gc, v.G - g0);
  const int64_t u0 = block * units;
  if (u0 >= v.n_munits) return;
  const int nu = (int)min((int64_t)units, v.n_munits - u0);
  const int64_t r0 = v.unit_off[u0];
  const int nr = (int)(v.unit_off[u0 + nu] - r0);
  GatherRun *runs = reinterpret_cast<GatherRun *>(msmem);
  float *P = reinterpret_cast<float *>(runs + nr);   // [3][run][group]
  const int nt = nr * gcount;
  {
    const int4 *src = reinterpret_cast<const int4 *>(v.gent + ch * v.gent_chunk + r0);
    for (int i = threadIdx.x; i < nr * (int)(sizeof(GatherRun) / 16); i += blockDim.x)
      copy16_async(reinterpret_cast<int4 *>(runs) + i, src + i);
    cp_async_commit();
    cp_async_wait<0>();
  }
  __syncthreads();
  chain_wait();   // the runs are the plan's; the state is the sweep's
  if (ch == 0 && block == 0 && threadIdx.x == 0)
    const_cast<double *>(a.scale)[3] = 1.0;   // the state is in this step's scale now
  // 1. the runs' sums
  const float *I = (const float *)a.I;
  {
    int r = (int)threadIdx.x / gcount, gi = (int)threadIdx.x - r * gcount;
    const int dr = (int)blockDim.x / gcount, dg = (int)blockDim.x - dr * gcount;
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {
      const GatherRun &run = runs[r];
      const int2 pc = *reinterpret_cast<const int2 *>(&run.pair);
      float P0 = 0.f, P1 = 0.f, P2 = 0.f;
      float c0[NP], c1[NP], c2[NP];
      const float *cf = v.fold + pc.x * kStride;
      load_fold<NP>(cf, c0);
      load_fold<NP>(cf + kRow, c1);
      load_fold<NP>(cf + 2 * kRow, c2);
#pragma unroll
      for (int k0 = 0; k0 < kRunSegments; k0 += kTogether) {
        float dv[kTogether][2][NP];
#pragma unroll
        for (int k = 0; k < kTogether; ++k) {
          const int4 s = run.seg[k0 + k];
          load_dev_if<NP>(k0 + k < pc.y, I + gather_slot(s.x, s.z, gi) * NP, dv[k][0]);
          load_dev_if<NP>(k0 + k < pc.y, I + gather_slot(s.y, s.w, gi) * NP, dv[k][1]);
        }
#pragma unroll
        for (int k = 0; k < kTogether; ++k) {   // an absent segment adds zeros (its area and values)
          const float af = run.area[k0 + k];
#pragma unroll
          for (int sense = 0; sense < 2; ++sense) {
            float S0 = 0.f, S1 = 0.f, S2 = 0.f;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
              S0 = fmaf(c0[p], dv[k][sense][p], S0);
              S1 = fmaf(c1[p], dv[k][sense][p], S1);
              S2 = fmaf(c2[p], dv[k][sense][p], S2);
            }
            P0 = fmaf(af, S0, P0);
            P1 = fmaf(sense ? -af : af, S1, P1);
            P2 = fmaf(af, S2, P2);
          }
        }
      }
      P[t] = P0;
      P[nt + t] = P1;
      P[2 * nt + t] = P2;
      r += dr;
      gi += dg;
      if (gi >= gcount) {
        gi -= gcount;
        ++r;
      }
    }
  }
  __syncthreads();
  // 2. the units' sums
  for (int k = threadIdx.x; k < nu * gcount; k += blockDim.x) {
    const int ul = k / gcount, gi = k - ul * gcount;
    const int64_t unit = u0 + ul;
    const int2 um = v.n_mmulti ? v.munit[unit] : make_int2((int)unit, 1);
    const int rb = (int)(v.unit_off[unit] - r0), re = (int)(v.unit_off[unit + 1] - r0);
    f32x2 hi[3] = {0, 0, 0}, lo[3] = {0, 0, 0};   // (E, Fx), (Fy, Nxx), (Nxy, Nyy)
#pragma unroll 4
    for (int r = rb; r < re; ++r) {
      const float2 cs = *reinterpret_cast<const float2 *>(&runs[r].cf);
      const int t = r * gcount + gi;
      const float P0 = P[t], P1 = P[nt + t], P2 = P[2 * nt + t];
      two_sum_add2(hi[0], lo[0], pack2(P0, cs.x * P1));
      two_sum_add2(hi[1], lo[1], mul2(pack2(cs.y, cs.x * cs.x), pack2(P1, P2)));
      two_sum_add2(hi[2], lo[2], mul2(pack2(cs.x * cs.y, cs.y * cs.y), pack2(P2, P2)));
    }
    // FP64 work here is per (cell, group), not per update: conversions by integer operations, one add per sum
    double D[kOutputs];
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      const float2 h = unpack2(hi[o]), l = unpack2(lo[o]);
      D[2 * o] = f32_to_f64(h.x) + f32_to_f64(l.x);
      D[2 * o + 1] = f32_to_f64(h.y) + f32_to_f64(l.y);
    }
    if (um.y == 1) {
      assemble_cell(v, a, um.x, g0 + gi, D);
    } else {
      double *ps = v.mscratch + (((int64_t)ch * v.n_munits + unit) * kOutputs) * L.gc + gi;
#pragma unroll
      for (int o = 0; o < kOutputs; ++o) ps[o * L.gc] = D[o];
    }
  }
}

// Split cells: the parts' partial sums added in part order (FP64), then assembled.  One thread per (split
// cell, group) of chunk ch, threads t0 ...
__device__ __forceinline__ void moments_combine_body(const PlanView &v, const SweepArgs &a, const Layout &L, int ch,
                                                     int64_t t0) {
  const int g0 = ch * L.gc;
  const int gcount = min(L.gc, v.G - g0);
  const int64_t t = t0 + threadIdx.x;
  if (t >= (int64_t)v.n_mmulti * gcount) return;
  const int m = (int)(t / gcount), gi = (int)(t - (int64_t)m * gcount);
  const int4 mc = v.mmulti[m];
  double D[kOutputs] = {0, 0, 0, 0, 0, 0};
  for (int k = 0; k < mc.z; ++k) {
    const double *ps = v.mscratch + (((int64_t)ch * v.n_munits + mc.y + k) * kOutputs) * L.gc + gi;
#pragma unroll
    for (int o = 0; o < kOutputs; ++o) D[o] += ps[o * L.gc];
  }
  assemble_cell(v, a, mc.x, g0 + gi, D);
}

__global__ void __launch_bounds__(128) moments_combine_kernel(PlanView v, SweepArgs a, Layout L) {
  chain_wait();
  moments_combine_body(v, a, L, blockIdx.y, (int64_t)blockIdx.x * blockDim.x);
}

__global__ void __launch_bounds__(128) moments_combine_batch_kernel(const BatchInst *inst, const int4 *map) {
  const int4 m = map[blockIdx.x];
  const BatchInst &b = inst[m.x];
  moments_combine_body(b.v, b.a, b.L, m.y, (int64_t)m.z * blockDim.x);
}

// (4 polar cosines: 72 registers; 64 spill, 3517 us a step at 512^2 x 17, 72 3437)
template <int NP>
__global__ void __launch_bounds__(kMomentBlock, moment_sm_blocks(NP)) moments_fp32_kernel(PlanView v, SweepArgs a, Layout L) {
  moments_fp32_body<NP>(v, a, L, blockIdx.y, blockIdx.x, v.munit_block[((int)blockIdx.y + 1) * L.gc > v.G]);
}

// Batched: block j is block map[j].z, of map[j].w units a block, of chunk map[j].y of instance map[j].x.
template <int NP>
__global__ void __launch_bounds__(kMomentBlock, moment_sm_blocks(NP))
    moments_fp32_batch_kernel(const BatchInst *inst, const int4 *map) {
  const int4 m = map[blockIdx.x];
  const BatchInst &b = inst[m.x];
  moments_fp32_body<NP>(b.v, b.a, b.L, m.y, m.z, m.w);
}

// Closure.  A block takes kRowCells cells, kRowGroups groups at a time: its threads load a (group, cell) each (cells
// fastest) and form what belongs to the group; the sums over groups are then taken from shared memory by one thread per
// (sum, cell), group by group in order.  One thread per cell, looping over the groups, left 64 blocks of serial chains of
// loads at 128^2 x 17 groups: 19.5 us back to back with its inputs in L2, so 11.2, bound by the FP64 pipe (one division a
// group and cell).  With one or two groups most of such a block has nothing to load, and one thread per cell is faster:
// 512^2 x 1 group 13.7 us for 21.5, 400^2 x 2 13.8 for 17.9 (one thread per cell at 5 groups 18.9 for 18.7).
constexpr int kRowCells = 32, kRowGroups = 8;

// f = N / (c E) per group (Eq. 7 with the cell averages of Eq. 15); <f>_E = sum_g N_g / (c sum_g E_g).
__global__ void __launch_bounds__(kRowCells *kRowGroups) closure_kernel(PlanView v, molc_moments m, double c, double *fxx,
                                                                        double *fxy, double *fyy, double *fgrey) {
  __shared__ double sm[4][kRowGroups][kRowCells];   // E, Nxx, Nxy, Nyy
  const int cl = threadIdx.x % kRowCells, gl = threadIdx.x / kRowCells;
  const int cell = blockIdx.x * kRowCells + cl;
  const bool in = cell < v.ncell;
  double sum = 0.0;
  for (int g0 = 0; g0 < v.G; g0 += kRowGroups) {
    if (in && g0 + gl < v.G) {
      const int64_t i = (int64_t)(g0 + gl) * v.ncell + cell;
      const double E = m.E[i], nxx = m.Nxx[i], nxy = m.Nxy[i], nyy = m.Nyy[i];
      const double inv = E > 0 ? 1.0 / (c * E) : 0.0;
      fxx[i] = nxx * inv;
      fxy[i] = nxy * inv;
      fyy[i] = nyy * inv;
      sm[0][gl][cl] = E;
      sm[1][gl][cl] = nxx;
      sm[2][gl][cl] = nxy;
      sm[3][gl][cl] = nyy;
    }
    if (!fgrey) continue;
    __syncthreads();
    if (gl < 4)
      for (int k = 0; k < min(kRowGroups, v.G - g0); ++k) sum += sm[gl][k][cl];
    __syncthreads();
  }
  if (!fgrey) return;
  if (gl < 4) sm[gl][0][cl] = sum;
  __syncthreads();
  if (gl == 0 || gl >= 4 || !in) return;
  const double se = sm[0][0][cl];
  const double inv = se > 0 ? 1.0 / (c * se) : 0.0;
  fgrey[(gl - 1) * (int64_t)v.ncell + cell] = sum * inv;
}

constexpr int kFewGroups = 2, kFewBlock = 128;
template <bool GREY>
__global__ void __launch_bounds__(kFewBlock) closure_few_kernel(PlanView v, molc_moments m, double c, double *fxx, double *fxy,
                                                                double *fyy, double *fgrey) {
  const int cell = blockIdx.x * kFewBlock + threadIdx.x;
  if (cell >= v.ncell) return;
  double se = 0, sxx = 0, sxy = 0, syy = 0;
  for (int g = 0; g < v.G; ++g) {
    const int64_t i = (int64_t)g * v.ncell + cell;
    const double E = m.E[i], nxx = m.Nxx[i], nxy = m.Nxy[i], nyy = m.Nyy[i];
    const double inv = E > 0 ? 1.0 / (c * E) : 0.0;
    fxx[i] = nxx * inv;
    fxy[i] = nxy * inv;
    fyy[i] = nyy * inv;
    if constexpr (GREY) {
      se += E;
      sxx += nxx;
      sxy += nxy;
      syy += nyy;
    }
  }
  if constexpr (!GREY) return;
  const double inv = se > 0 ? 1.0 / (c * se) : 0.0;
  fgrey[cell] = sxx * inv;
  fgrey[v.ncell + cell] = sxy * inv;
  fgrey[2 * (int64_t)v.ncell + cell] = syy * inv;
}

// Grey-problem coefficients (Eqs. 8-9), all in FP64: <kappa>_E, <kappa>_B, the flux-weighted
// K_R = diag(<kappa>_|Fx|, <kappa>_|Fy|) and eta = sum_g (kappa_g - K_R) F_g / sum_g E_g.  The results are written last: they
// may lie over an input.
// One thread per cell with the loads of kGreyGroups groups in flight, in blocks of one warp so that small grids reach all
// SMs; the FP64 pipe bounds it (twelve operations a group and cell).  Where that leaves less than a warp an SM the groups
// are shared out too (grey_small_kernel).  Back to back, one thread per cell, blocks of cells x groups: 64^2 x 17 groups
// 11.2 and 7.1 us (13.6 with one group's loads in flight), 100^2 x 37 21.6 and 26.9, 128^2 x 17 11.8 and 17.5 (13.4),
// 512^2 x 17 126 and 211 (125), 512^2 x 1 44 and 49 (44).
constexpr int kGreyBlock = 32, kGreyGroups = 4;
__global__ void __launch_bounds__(kGreyBlock) grey_kernel(PlanView v, molc_moments m, const double *kappa, const double *B,
                                                          double *out) {
  const int cell = blockIdx.x * kGreyBlock + threadIdx.x;
  if (cell >= v.ncell) return;
  const int64_t n = v.ncell;
  double se = 0, ske = 0, sb = 0, skb = 0, sfx = 0, skfx = 0, sfy = 0, skfy = 0;
  for (int g0 = 0; g0 < v.G; g0 += kGreyGroups) {
    double k[kGreyGroups], E[kGreyGroups], b[kGreyGroups], fx[kGreyGroups], fy[kGreyGroups];
#pragma unroll
    for (int j = 0; j < kGreyGroups; ++j) {
      if (g0 + j >= v.G) break;
      const int64_t i = (int64_t)(g0 + j) * n + cell;
      k[j] = kappa[i];
      E[j] = m.E[i];
      b[j] = B[i];
      fx[j] = fabs(m.Fx[i]);
      fy[j] = fabs(m.Fy[i]);
    }
#pragma unroll
    for (int j = 0; j < kGreyGroups; ++j) {
      if (g0 + j >= v.G) break;
      se += E[j];
      ske = fma(k[j], E[j], ske);
      sb += b[j];
      skb = fma(k[j], b[j], skb);
      sfx += fx[j];
      skfx = fma(k[j], fx[j], skfx);
      sfy += fy[j];
      skfy = fma(k[j], fy[j], skfy);
    }
  }
  const double kE = se > 0 ? ske / se : 0.0, kB = sb > 0 ? skb / sb : 0.0;
  const double kx = sfx > 0 ? skfx / sfx : 0.0, ky = sfy > 0 ? skfy / sfy : 0.0;
  double ex = 0, ey = 0;
  for (int g0 = 0; g0 < v.G; g0 += kGreyGroups) {
    double k[kGreyGroups], fx[kGreyGroups], fy[kGreyGroups];
#pragma unroll
    for (int j = 0; j < kGreyGroups; ++j) {
      if (g0 + j >= v.G) break;
      const int64_t i = (int64_t)(g0 + j) * n + cell;
      k[j] = kappa[i];
      fx[j] = m.Fx[i];
      fy[j] = m.Fy[i];
    }
#pragma unroll
    for (int j = 0; j < kGreyGroups; ++j) {
      if (g0 + j >= v.G) break;
      ex = fma(k[j] - kx, fx[j], ex);
      ey = fma(k[j] - ky, fy[j], ey);
    }
  }
  out[cell] = kE;
  out[n + cell] = kB;
  out[2 * n + cell] = kx;
  out[3 * n + cell] = ky;
  out[4 * n + cell] = se > 0 ? ex / se : 0.0;
  out[5 * n + cell] = se > 0 ? ey / se : 0.0;
}

// The same with a (group, cell) loaded by a thread of its own, as in closure_kernel.
__global__ void __launch_bounds__(kRowCells *kRowGroups) grey_small_kernel(PlanView v, molc_moments m, const double *kappa,
                                                                           const double *B, double *out) {
  __shared__ double sm[5][kRowGroups][kRowCells];   // kappa, E, B, Fx, Fy
  const int cl = threadIdx.x % kRowCells, gl = threadIdx.x / kRowCells;
  const int cell = blockIdx.x * kRowCells + cl;
  const bool in = cell < v.ncell;
  const int64_t n = v.ncell;
  // sums 2 x and 2 x + 1 of thread row gl: of E, B, |Fx|, |Fy| and of kappa times it
  const int x = 1 + gl / 2;
  double sum = 0.0;
  for (int g0 = 0; g0 < v.G; g0 += kRowGroups) {
    if (in && g0 + gl < v.G) {
      const int64_t i = (int64_t)(g0 + gl) * n + cell;
      sm[0][gl][cl] = kappa[i];
      sm[1][gl][cl] = m.E[i];
      sm[2][gl][cl] = B[i];
      sm[3][gl][cl] = fabs(m.Fx[i]);
      sm[4][gl][cl] = fabs(m.Fy[i]);
    }
    __syncthreads();
    for (int k = 0; k < min(kRowGroups, v.G - g0); ++k)
      sum = gl & 1 ? fma(sm[0][k][cl], sm[x][k][cl], sum) : sum + sm[x][k][cl];
    __syncthreads();
  }
  sm[0][gl][cl] = sum;
  __syncthreads();
  double mean = 0.0;   // of rows 0 to 3: <kappa>_E, <kappa>_B, K_Rx, K_Ry
  if (gl < 4) {
    const double s = sm[0][2 * gl][cl];
    mean = s > 0 ? sm[0][2 * gl + 1][cl] / s : 0.0;
  }
  const double se = sm[0][0][cl];
  double eta = 0.0;   // rows 2 and 3: sum_g (kappa_g - K_R) F_g
  for (int g0 = 0; g0 < v.G; g0 += kRowGroups) {
    __syncthreads();
    if (in && g0 + gl < v.G) {
      const int64_t i = (int64_t)(g0 + gl) * n + cell;
      sm[0][gl][cl] = kappa[i];
      sm[3][gl][cl] = m.Fx[i];
      sm[4][gl][cl] = m.Fy[i];
    }
    __syncthreads();
    if (gl == 2 || gl == 3)
      for (int k = 0; k < min(kRowGroups, v.G - g0); ++k) eta = fma(sm[0][k][cl] - mean, sm[gl + 1][k][cl], eta);
  }
  if (!in || gl >= 4) return;
  out[gl * n + cell] = mean;
  if (gl >= 2) out[(gl + 2) * n + cell] = se > 0 ? eta / se : 0.0;
}

// Canonical segment averages <-> deviation state, Ibar = B_ref(cell) + delta: one block per (track, sense).  The
// canonical rows of one (track, sense, polar cosine) are contiguous, [step][selected group], so consecutive threads
// take consecutive (step, group) pairs and, for each, the NP adjacent deviations of the state (a block reads runs of
// groups x NP values and writes NP contiguous streams).  One thread per state row, looping over polar cosines and
// groups, had every lane on rows of its own: 64^2 x 17 groups, 4 x 32 directions, h/4 (4.6e7 values, 0.55 GB)
// 565 us either way; so it is 135 us out and 159 us in.  That is bound by the FP64 pipe (one addition a value; the
// power-of-two scalings and the conversions are integer operations), with DRAM at 3.5 TB/s next.
// One thread's elements of a walk, (step, group) by (step, group): f(step, group).
template <class F>
__device__ __forceinline__ void for_walk(int nseg, int g_count, F f) {
  int s = (int)threadIdx.x / g_count, gi = (int)threadIdx.x - s * g_count;
  const int ds = (int)blockDim.x / g_count, dg = (int)blockDim.x - ds * g_count;
  for (; s < nseg; s += ds) {
    f(s, gi);
    gi += dg;
    if (gi >= g_count) {
      gi -= g_count;
      ++s;
    }
  }
}

template <int NP, bool TO_CANON>
__global__ void __launch_bounds__(128) intensity_copy_fp32_kernel(PlanView v, Layout L, float *I, const double *Bref,
                                                                  const double *scale, int g_begin, int g_count,
                                                                  double *canon) {
  // 1/scale and scale are powers of two
  const double sc = scale[0], is = scale[1];
  const int k_out = exponent_of(is), k_in = exponent_of(sc);
  const TrackDev tr = v.tracks[blockIdx.x >> 1];
  const int sense = blockIdx.x & 1;
  const int pos = sense ? tr.pos[1] : tr.pos[0];
  const int64_t cs = sense ? tr.canon_minus : tr.canon_plus;
  double *cv[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const PolarDev &pd = v.polar[tr.pair * NP + p];
    cv[p] = canon + (v.dir_seg_off[sense ? pd.dir_minus : pd.dir_plus] + cs) * g_count;
  }
  const int *cells = v.seg_cell + (sense ? tr.seg_off + tr.nseg - 1 : tr.seg_off);
  auto element = [&](int s, int gi, bool fast) {
    const int g = g_begin + gi, ch = g / L.gc, gl = g - ch * L.gc, gcount = min(L.gc, v.G - ch * L.gc);
    float *el = I + bundle_index(v.boff, (int64_t)ch * 2 * v.n_tracks * L.gc + (int64_t)pos * gcount + gl, s, NP);
    const double br = Bref[(int64_t)g * v.ncell + cells[sense ? -s : s]];
    const int64_t o = (int64_t)s * g_count + gi;
    float x[NP];
    if constexpr (TO_CANON) {
      load_dev_cg<NP>(el, x);
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        __stcs(cv[p] + o, br + (fast ? scaled_to_double(x[p], k_out) : (double)x[p] * is));
      }
    } else {
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const double y = __ldcs(cv[p] + o) - br;
        x[p] = fast ? scaled_to_float(y, k_in) : (float)(y * sc);
      }
#pragma unroll
      for (int p = 0; p < NP; ++p) el[p] = x[p];
    }
  };
  if (abs(k_out) < 1023 && abs(k_in) < 1023)
    for_walk(tr.nseg, g_count, [&](int s, int gi) { element(s, gi, true); });
  else   // a scale outside the normal range
    for_walk(tr.nseg, g_count, [&](int s, int gi) { element(s, gi, false); });
}

// The FP64 state: rows (track, sense, step) of [G][NP].
template <bool TO_CANON>
__global__ void __launch_bounds__(128) intensity_copy_fp64_kernel(PlanView v, double *I, const double *Bref, int g_begin,
                                                                  int g_count, double *canon) {
  const int NP = v.n_polar;
  const TrackDev tr = v.tracks[blockIdx.x >> 1];
  const int sense = blockIdx.x & 1;
  const int64_t cs = sense ? tr.canon_minus : tr.canon_plus;
  const int *cells = v.seg_cell + (sense ? tr.seg_off + tr.nseg - 1 : tr.seg_off);
  for_walk(tr.nseg, g_count, [&](int s, int gi) {
    const int g = g_begin + gi;
    double *el = I + ((2 * tr.seg_off + (int64_t)sense * tr.nseg + s) * v.G + g) * NP;
    const double br = Bref[(int64_t)g * v.ncell + cells[sense ? -s : s]];
    for (int p = 0; p < NP; ++p) {
      const PolarDev &pd = v.polar[tr.pair * NP + p];
      double *cv = canon + (v.dir_seg_off[sense ? pd.dir_minus : pd.dir_plus] + cs + s) * g_count + gi;
      if constexpr (TO_CANON)
        __stcs(cv, br + el[p]);
      else
        el[p] = __ldcs(cv) - br;
    }
  });
}

// max over finite non-negative B of the IEEE bits (ordered like the values for x >= 0)
__global__ void max_bits_kernel(const double *B, int64_t n, unsigned long long *mx) {
  unsigned long long m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double b = B[i];
    if (b >= 0.0 && isfinite(b)) m = max(m, (unsigned long long)__double_as_longlong(b));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
  if ((threadIdx.x & 31) == 0 && m) atomicMax(mx, m);
}

// scale = 2^(100 - e) with max B = f 2^e, f in [1/2, 1) (2^100 if max B = 0); 1 for FP64 states.
__global__ void set_scale_kernel(const unsigned long long *mx, double *header, int fp32) {
  double s = 1.0;
  if (fp32) {
    const double m = __longlong_as_double((long long)*mx);
    int e = 0;
    if (m > 0.0) frexp(m, &e);
    s = ldexp(1.0, kScaleTargetExp - e);
  }
  header[0] = s;
  header[1] = 1.0 / s;
  header[3] = 1.0;
  reinterpret_cast<unsigned long long *>(header)[2] = 0;   // the sweep-time reduction starts from zero
  reinterpret_cast<unsigned int *>(header + 4)[0] = 0;     // and with no block counted
}

// Sweep-time scale of an FP32 state: the scale follows max(B, boundary) so that the largest scaled intensity
// stays near 2^100.  It is kept while that maximum, scaled, has its exponent in [93, 108]; otherwise it is reset
// to 2^(100 - e), max = f 2^e.  header[3] = new scale / old scale (a power of two) is the factor by which this
// step's sweep multiplies the stored deviations as it reads them; the moment kernel sets it back to 1.
__device__ __forceinline__ void update_scale(unsigned long long mbits, double *header) {
  const double m = __longlong_as_double((long long)mbits);
  const double s = header[0];
  double f = 1.0;
  if (m > 0.0 && isfinite(m)) {
    int em = 0, es = 0;
    frexp(m, &em);
    frexp(s, &es);
    const int e = em + es - 1;   // exponent of m * s (s is a power of two)
    if (e < 93 || e > 108) {
      const double sn = ldexp(1.0, kScaleTargetExp - em);
      f = sn / s;
      header[0] = sn;
      header[1] = 1.0 / sn;
    }
  }
  header[3] = f;
}

// One launch: every block folds its share of B (block 0 also the boundary) into header[2] by atomicMax; the
// last block to finish (counted in header[4]) updates the scale and leaves both words at zero for the next call.
__global__ void __launch_bounds__(256) update_scale_kernel(const double *B, int64_t n, const double *bnd, int nb,
                                                         double *header) {
  __shared__ unsigned long long red[8];
  chain_next();
  unsigned long long *mx = reinterpret_cast<unsigned long long *>(header + 2);
  unsigned int *cnt = reinterpret_cast<unsigned int *>(header + 4);
  unsigned long long m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double x = B[i];
    if (x >= 0.0 && isfinite(x)) m = max(m, (unsigned long long)__double_as_longlong(x));
  }
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
      const double x = bnd[i];
      if (x >= 0.0 && isfinite(x)) m = max(m, (unsigned long long)__double_as_longlong(x));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(kFull, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, red[w]);
    if (m) atomicMax(mx, m);
    __threadfence();
    if (atomicAdd(cnt, 1u) == gridDim.x - 1) {   // last block: every other block's maximum is in place
      __threadfence();
      const unsigned long long all = atomicMax(mx, 0ull);
      update_scale(all, header);
      *mx = 0;
      *cnt = 0;
    }
  }
}

// Batched, several blocks per instance: map[block] = {instance, block of the instance, blocks of the instance, 0}.
// Each block folds its share of the instance's B (its block 0 also the boundary) into the instance's header[2] by
// atomicMax; the last of the instance's blocks (counted in header[4]) updates that instance's scale, as
// update_scale_kernel does for one plan.
template <class Inst>
__global__ void __launch_bounds__(256) update_scale_map_kernel(const Inst *inst, const int4 *map) {
  __shared__ unsigned long long red[8];
  const int4 m = map[blockIdx.x];
  const Inst &b = inst[m.x];
  double *header = const_cast<double *>(b.a.scale);
  unsigned long long *mx = reinterpret_cast<unsigned long long *>(header + 2);
  unsigned int *cnt = reinterpret_cast<unsigned int *>(header + 4);
  const int64_t n = (int64_t)b.v.G * b.v.ncell;
  unsigned long long v = 0;
  for (int64_t i = (int64_t)m.y * blockDim.x + threadIdx.x; i < n; i += (int64_t)m.z * blockDim.x) {
    const double x = b.a.B[i];
    if (x >= 0.0 && isfinite(x)) v = max(v, (unsigned long long)__double_as_longlong(x));
  }
  if (m.y == 0)
    for (int i = threadIdx.x; i < 4 * b.v.G; i += blockDim.x) {
      const double x = b.a.bnd[i];
      if (x >= 0.0 && isfinite(x)) v = max(v, (unsigned long long)__double_as_longlong(x));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = max(v, red[w]);
    if (v) atomicMax(mx, v);
    __threadfence();
    if (atomicAdd(cnt, 1u) == (unsigned)m.z - 1) {   // last block of this instance
      __threadfence();
      const unsigned long long all = atomicMax(mx, 0ull);
      update_scale(all, header);
      *mx = 0;
      *cnt = 0;
    }
  }
}

int grid_for(int64_t n, int block) {
  int64_t b = (n + block - 1) / block;
  if (b < 1) b = 1;
  if (b > 152 * 64) b = 152 * 64;
  return (int)b;
}

}  // namespace

// Blocks of the preparation over one chunk; which links of an FP32 step are chained.
static int prep_blocks(const PlanView &v) { return std::min((v.ncell + kPrepCells - 1) / kPrepCells, 152 * 16); }
static bool chained(const PlanView &v) {
  return few_walks(v) && (int64_t)prep_blocks(v) * layout_for(v, MOLC_FP32).n_chunks <= 152 * 4;
}
static bool sweep_chained(const PlanView &v) {
  return few_walks(v) && (int64_t)prep_blocks(v) * layout_for(v, MOLC_FP32).n_chunks <= (v.n_polar <= 4 ? 152 : 76);
}

cudaError_t launch_prep(const PlanView &v, const SweepArgs &a, cudaStream_t st) {
  const Layout L = layout_for(v, MOLC_FP32);
  if (L.gc > 32 || L.n_chunks > 65535) return cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)prep_blocks(v), (unsigned)L.n_chunks);
  return launch_chained(chained(v), prep_kernel, grid, 128, 0, st, v, a, L);
}

template <int D>
static cudaError_t sweep_fp32_depth(const PlanView &v, const SweepArgs &a, const Layout &L, dim3 grid,
                                    cudaStream_t st) {
  switch (v.n_polar) {
    case 1: return launch_chained(sweep_chained(v), sweep_fp32_kernel<1, D>, grid, kSweepBlock, 0, st, v, a, L);
    case 2: return launch_chained(sweep_chained(v), sweep_fp32_kernel<2, D>, grid, kSweepBlock, 0, st, v, a, L);
    case 3: return launch_chained(sweep_chained(v), sweep_fp32_kernel<3, D>, grid, kSweepBlock, 0, st, v, a, L);
    case 4: return launch_chained(sweep_chained(v), sweep_fp32_kernel<4, D>, grid, kSweepBlock, 0, st, v, a, L);
    case 5: return launch_chained(sweep_chained(v), sweep_fp32_kernel<5, D>, grid, kSweepBlock, 0, st, v, a, L);
    case 6: return launch_chained(sweep_chained(v), sweep_fp32_kernel<6, D>, grid, kSweepBlock, 0, st, v, a, L);
    case 7: return launch_chained(sweep_chained(v), sweep_fp32_kernel<7, D>, grid, kSweepBlock, 0, st, v, a, L);
    case 8: return launch_chained(sweep_chained(v), sweep_fp32_kernel<8, D>, grid, kSweepBlock, 0, st, v, a, L);
    default: return cudaErrorInvalidValue;
  }
}

template <int EXTRA>
cudaError_t sweep_fp32_extra(const PlanView &v, const SweepArgs &a, const Layout &L, dim3 grid, cudaStream_t st) {
  switch (v.n_polar) {
    case 1: return launch_chained(sweep_chained(v), sweep_fp32_kernel<1, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    case 2: return launch_chained(sweep_chained(v), sweep_fp32_kernel<2, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    case 3: return launch_chained(sweep_chained(v), sweep_fp32_kernel<3, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    case 4: return launch_chained(sweep_chained(v), sweep_fp32_kernel<4, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    case 5: return launch_chained(sweep_chained(v), sweep_fp32_kernel<5, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    case 6: return launch_chained(sweep_chained(v), sweep_fp32_kernel<6, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    case 7: return launch_chained(sweep_chained(v), sweep_fp32_kernel<7, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    case 8: return launch_chained(sweep_chained(v), sweep_fp32_kernel<8, 4, EXTRA>, grid, kSweepBlock, 0, st, v, a, L);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_sweep_fp32(const PlanView &v, const SweepArgs &a, cudaStream_t st) {
  const Layout L = layout_for(v, MOLC_FP32);
  const int64_t blocks = (a.n_items + kSweepBlock - 1) / kSweepBlock;
  if (blocks > 0x7fffffff) return cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)blocks);
  if (v.facc) return sweep_fp32_extra<kSweepFaces>(v, a, L, grid, st);       // face reductions, depth 4
  if (v.balance) return sweep_fp32_extra<kSweepBalance>(v, a, L, grid, st);  // per-ray balance check, depth 4
  switch (v.sweep_depth) {
    case 3: return sweep_fp32_depth<3>(v, a, L, grid, st);
    case 4: return sweep_fp32_depth<4>(v, a, L, grid, st);
    case 6: return sweep_fp32_depth<6>(v, a, L, grid, st);
    default: return cudaErrorInvalidValue;
  }
}

// A kernel's limit of dynamic shared memory is the whole process's: it is set to the most that any plan's gather takes, the
// same by every thread, not to this plan's size, which another thread could lower before the launch.
template <class K>
static cudaError_t allow_moment_smem(K *kernel) {
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)moment_smem(kPartSegments, 32));
  if (e != cudaSuccess) cudaGetLastError();   // reported here, not by the next launch
  return e;
}

cudaError_t launch_moments_fp32(const PlanView &v, const SweepArgs &a, cudaStream_t st) {
  const Layout L = layout_for(v, MOLC_FP32);
  const int64_t blocks = moment_blocks(v, v.G >= L.gc * L.n_chunks ? v.munit_block[0] : std::min(v.munit_block[0], v.munit_block[1]));
  if (blocks > 0x7fffffff || L.n_chunks > 65535) return cudaErrorInvalidConfiguration;
  const dim3 grid((unsigned)blocks, (unsigned)L.n_chunks);
  const size_t smem = v.msmem;
  cudaError_t e = cudaSuccess;
  switch (v.n_polar) {
#define MOLC_MOMENTS(NP)                                                                                          \
  case NP:                                                                                                        \
    if (smem > 48 * 1024) e = allow_moment_smem(moments_fp32_kernel<NP>);                                        \
    if (e == cudaSuccess) e = launch_chained(chained(v), moments_fp32_kernel<NP>, grid, kMomentBlock, smem, st, v, a, L);  \
    break;
    MOLC_MOMENTS(1)
    MOLC_MOMENTS(2)
    MOLC_MOMENTS(3)
    MOLC_MOMENTS(4)
    MOLC_MOMENTS(5)
    MOLC_MOMENTS(6)
    MOLC_MOMENTS(7)
    MOLC_MOMENTS(8)
#undef MOLC_MOMENTS
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess || v.n_mmulti == 0) return e;
  const dim3 cgrid((unsigned)(((int64_t)v.n_mmulti * L.gc + 127) / 128), (unsigned)L.n_chunks);
  return launch_chained(chained(v), moments_combine_kernel, cgrid, 128, 0, st, v, a, L);
}

// Face moments from the face sums: E_f = D is / (c |f|), F_f, N_f = sums is / |f|; is = 1/scale of the state
// (1 for FP64), |f| = hy on x-faces, hx on y-faces.  A block turns `rows` faces x up to kFaceGroups groups of
// [face][6][gc] sums into [g][face] outputs through shared memory: reading them a (face, group) per thread, faces
// fastest, every lane had lines of its own.  The two divisors are taken once a block.
// With few groups a block takes more faces, so that its threads have sums to read.  Back to back, one thread per (face,
// group), then so (16 faces a block whatever the groups): 128^2 x 17 groups 25.7 us, 15.7 (16.0); 512^2 x 1 23.6, 14.9 (156);
// 256^2 x 8 46.3, 26.7 (55.2); 64^2 x 4 4.2, 3.7 (6.1); 512^2 x 17 1098, 244 (272).
constexpr int kFaceRows = 16, kFaceGroups = 32;
__global__ void __launch_bounds__(256) face_moments_kernel(PlanView v, Layout L, const double *scale, double c, double hx,
                                                           double hy, int rows, molc_moments out) {
  __shared__ double sm[kOutputs * kFaceGroups * (kFaceRows + 1)];   // [output][group][rows + 1]
  __shared__ double factor[2][2];   // x-faces, y-faces: is / |f|, is / (c |f|)
  const int face_blocks = (v.n_faces + rows - 1) / rows, slices = (L.gc + kFaceGroups - 1) / kFaceGroups;
  const int row = blockIdx.x / face_blocks, ch = row / slices, gs = (row - ch * slices) * kFaceGroups;
  const int ng = min(kFaceGroups, min(L.gc, v.G - ch * L.gc) - gs);
  if (ng <= 0) return;
  const int f0 = (blockIdx.x - row * face_blocks) * rows, nf = min(rows, v.n_faces - f0);
  if (threadIdx.x < 2) {
    const double r = (scale ? scale[1] : 1.0) / (threadIdx.x ? hx : hy);
    factor[threadIdx.x][0] = r;
    factor[threadIdx.x][1] = r / c;
  }
  const double *fa = v.facc + ((int64_t)ch * v.n_faces + f0) * kOutputs * L.gc + gs;
  const int pitch = rows + 1;
  for (int k = threadIdx.x; k < nf * kOutputs * ng; k += blockDim.x) {
    const int fo = k / ng, gl = k - fo * ng;
    sm[((fo % kOutputs) * ng + gl) * pitch + fo / kOutputs] = fa[(int64_t)fo * L.gc + gl];
  }
  __syncthreads();
  const int nxf = (v.nx + 1) * v.ny;
  for (int k = threadIdx.x; k < ng * nf; k += blockDim.x) {
    const int gl = k / nf, fl = k - gl * nf;
    const int64_t i = (int64_t)(ch * L.gc + gs + gl) * v.n_faces + f0 + fl;
    const double *r = factor[f0 + fl < nxf ? 0 : 1], *x = sm + gl * pitch + fl;
    out.E[i] = x[0] * r[1];
    out.Fx[i] = x[ng * pitch] * r[0];
    out.Fy[i] = x[2 * ng * pitch] * r[0];
    out.Nxx[i] = x[3 * ng * pitch] * r[0];
    out.Nxy[i] = x[4 * ng * pitch] * r[0];
    out.Nyy[i] = x[5 * ng * pitch] * r[0];
  }
}

cudaError_t launch_face_moments(const PlanView &v, molc_precision prec, const double *scale, double c,
                                const molc_moments &out, cudaStream_t st) {
  const Layout L = layout_for(v, prec);
  const int64_t slices = (int64_t)L.n_chunks * ((L.gc + kFaceGroups - 1) / kFaceGroups);
  // as many faces as fill the block's shared memory with few groups, but no fewer blocks than 4 an SM
  int rows = kFaceRows;
  while (2 * rows * std::min(L.gc, kFaceGroups) <= kFaceRows * kFaceGroups && v.n_faces / (2 * rows) * slices >= 152 * 4) rows *= 2;
  const int64_t blocks = (v.n_faces + rows - 1) / rows * slices;
  if (blocks > 0x7fffffff) return cudaErrorInvalidConfiguration;   // more sums than device memory holds
  face_moments_kernel<<<(unsigned)blocks, 256, 0, st>>>(v, L, scale, c, v.hx, v.hy, rows, out);
  return cudaGetLastError();
}

cudaError_t launch_grey(const PlanView &v, const molc_moments &m, const double *kappa, const double *B,
                        double *out, cudaStream_t st) {
  if (v.ncell <= 152 * kGreyBlock)
    grey_small_kernel<<<(v.ncell + kRowCells - 1) / kRowCells, kRowCells * kRowGroups, 0, st>>>(v, m, kappa, B, out);
  else
    grey_kernel<<<(v.ncell + kGreyBlock - 1) / kGreyBlock, kGreyBlock, 0, st>>>(v, m, kappa, B, out);
  return cudaGetLastError();
}

cudaError_t launch_closure(const PlanView &v, const molc_moments &m, double c, double *fxx, double *fxy,
                           double *fyy, double *f_grey, cudaStream_t st) {
  const unsigned few = (unsigned)((v.ncell + kFewBlock - 1) / kFewBlock);
  if (v.G > kFewGroups)
    closure_kernel<<<(v.ncell + kRowCells - 1) / kRowCells, kRowCells * kRowGroups, 0, st>>>(v, m, c, fxx, fxy, fyy, f_grey);
  else if (f_grey)
    closure_few_kernel<true><<<few, kFewBlock, 0, st>>>(v, m, c, fxx, fxy, fyy, f_grey);
  else
    closure_few_kernel<false><<<few, kFewBlock, 0, st>>>(v, m, c, fxx, fxy, fyy, f_grey);
  return cudaGetLastError();
}

cudaError_t launch_update_scale(const PlanView &v, const double *B, const double *bnd, double *header,
                                cudaStream_t st) {
  const int64_t n = (int64_t)v.G * v.ncell;
  update_scale_kernel<<<std::min(grid_for(n, 256), 152 * 4), 256, 0, st>>>(B, n, bnd, 4 * v.G, header);
  return cudaGetLastError();
}

cudaError_t launch_update_scale_map(const BatchInst *inst, const TileInst *tinst, const int4 *map, int blocks,
                                    cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  if (tinst)
    update_scale_map_kernel<TileInst><<<blocks, 256, 0, st>>>(tinst, map);
  else
    update_scale_map_kernel<BatchInst><<<blocks, 256, 0, st>>>(inst, map);
  return cudaGetLastError();
}

cudaError_t launch_prep_batch(const BatchInst *inst, const int4 *map, int blocks, cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  return launch_chained(false, prep_batch_kernel, blocks, 128, 0, st, inst, map);
}

template <int D>
static cudaError_t sweep_fp32_batch_depth(const BatchInst *inst, const int2 *map, int blocks, int n_polar,
                                          cudaStream_t st) {
  switch (n_polar) {
    case 1: return launch_chained(false, sweep_fp32_batch_kernel<1, D>, blocks, kSweepBlock, 0, st, inst, map);
    case 2: return launch_chained(false, sweep_fp32_batch_kernel<2, D>, blocks, kSweepBlock, 0, st, inst, map);
    case 3: return launch_chained(false, sweep_fp32_batch_kernel<3, D>, blocks, kSweepBlock, 0, st, inst, map);
    case 4: return launch_chained(false, sweep_fp32_batch_kernel<4, D>, blocks, kSweepBlock, 0, st, inst, map);
    case 5: return launch_chained(false, sweep_fp32_batch_kernel<5, D>, blocks, kSweepBlock, 0, st, inst, map);
    case 6: return launch_chained(false, sweep_fp32_batch_kernel<6, D>, blocks, kSweepBlock, 0, st, inst, map);
    case 7: return launch_chained(false, sweep_fp32_batch_kernel<7, D>, blocks, kSweepBlock, 0, st, inst, map);
    case 8: return launch_chained(false, sweep_fp32_batch_kernel<8, D>, blocks, kSweepBlock, 0, st, inst, map);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_sweep_fp32_batch(const BatchInst *inst, const int2 *map, int blocks, int n_polar, int depth,
                                    cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  switch (depth) {
    case 3: return sweep_fp32_batch_depth<3>(inst, map, blocks, n_polar, st);
    case 4: return sweep_fp32_batch_depth<4>(inst, map, blocks, n_polar, st);
    case 6: return sweep_fp32_batch_depth<6>(inst, map, blocks, n_polar, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_moments_fp32_batch(const BatchInst *inst, const int4 *map, int blocks, int n_polar,
                                      size_t smem, cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  cudaError_t e = cudaSuccess;
  switch (n_polar) {
#define MOLC_MOMENTS_B(NP)                                                                                          \
  case NP:                                                                                                        \
    if (smem > 48 * 1024) e = allow_moment_smem(moments_fp32_batch_kernel<NP>);                                     \
    if (e == cudaSuccess) e = launch_chained(false, moments_fp32_batch_kernel<NP>, blocks, kMomentBlock, smem, st, inst, map);  \
    break;
    MOLC_MOMENTS_B(1)
    MOLC_MOMENTS_B(2)
    MOLC_MOMENTS_B(3)
    MOLC_MOMENTS_B(4)
    MOLC_MOMENTS_B(5)
    MOLC_MOMENTS_B(6)
    MOLC_MOMENTS_B(7)
    MOLC_MOMENTS_B(8)
#undef MOLC_MOMENTS_B
    default: return cudaErrorInvalidValue;
  }
  return e;
}

cudaError_t launch_moments_combine_batch(const BatchInst *inst, const int4 *map, int blocks, cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  return launch_chained(false, moments_combine_batch_kernel, blocks, 128, 0, st, inst, map);
}


cudaError_t launch_intensity_copy(const PlanView &v, molc_precision prec, void *I, const double *Bref,
                                  const double *scale, int g_begin, int g_count, double *canon, bool to_canon,
                                  cudaStream_t st) {
  const Layout L = layout_for(v, prec);
  if (v.n_tracks > 0x3fffffff) return cudaErrorInvalidConfiguration;
  const unsigned blocks = (unsigned)(2 * v.n_tracks);
  if (prec == MOLC_FP64) {
    if (to_canon)
      intensity_copy_fp64_kernel<true><<<blocks, 128, 0, st>>>(v, (double *)I, Bref, g_begin, g_count, canon);
    else
      intensity_copy_fp64_kernel<false><<<blocks, 128, 0, st>>>(v, (double *)I, Bref, g_begin, g_count, canon);
    return cudaGetLastError();
  }
  switch (v.n_polar) {
#define MOLC_COPY(NP)                                                                                                  \
  case NP:                                                                                                             \
    if (to_canon)                                                                                                      \
      intensity_copy_fp32_kernel<NP, true><<<blocks, 128, 0, st>>>(v, L, (float *)I, Bref, scale, g_begin, g_count, canon); \
    else                                                                                                               \
      intensity_copy_fp32_kernel<NP, false><<<blocks, 128, 0, st>>>(v, L, (float *)I, Bref, scale, g_begin, g_count, canon); \
    break;
    MOLC_COPY(1)
    MOLC_COPY(2)
    MOLC_COPY(3)
    MOLC_COPY(4)
    MOLC_COPY(5)
    MOLC_COPY(6)
    MOLC_COPY(7)
    MOLC_COPY(8)
#undef MOLC_COPY
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_balance_scale(const PlanView &v, const double *B, const double *bnd, cudaStream_t st) {
  unsigned long long *mx = v.balance + 1;
  max_bits_kernel<<<grid_for((int64_t)v.G * v.ncell, 256), 256, 0, st>>>(B, (int64_t)v.G * v.ncell, mx);
  max_bits_kernel<<<1, 256, 0, st>>>(bnd, 4 * (int64_t)v.G, mx);
  return cudaGetLastError();
}

cudaError_t launch_set_scale(const PlanView &v, molc_precision prec, const double *B, double *header,
                             cudaStream_t st) {
  unsigned long long *mx = reinterpret_cast<unsigned long long *>(header + 2);
  cudaError_t e = cudaMemsetAsync(mx, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  max_bits_kernel<<<grid_for((int64_t)v.G * v.ncell, 256), 256, 0, st>>>(B, (int64_t)v.G * v.ncell, mx);
  set_scale_kernel<<<1, 1, 0, st>>>(mx, header, prec == MOLC_FP32);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------------------
// FP64 FMA throughput of this GPU (the bound of the plain FP64 sweep, whose intensity updates and polar folds are FP64): every thread runs kFmaChains independent chains of kFmaIters dependent FMAs, so the FP64
// pipe, not latency, limits the rate.  The chains' sum is compared with a value it never takes and stored, if it
// did, to a static device variable, so that the work cannot be dropped and no pointer is needed.
// ---------------------------------------------------------------------------------------------------------
constexpr int kFmaChains = 8, kFmaIters = 4096;
__device__ double g_fma_sink;
__global__ void __launch_bounds__(256) fp64_fma_kernel(double a, double b) {
  double x[kFmaChains];
#pragma unroll
  for (int k = 0; k < kFmaChains; ++k) x[k] = threadIdx.x * 1e-3 + k;
  for (int i = 0; i < kFmaIters; ++i) {
#pragma unroll
    for (int k = 0; k < kFmaChains; ++k) x[k] = fma(x[k], a, b);
  }
  double s = 0;
#pragma unroll
  for (int k = 0; k < kFmaChains; ++k) s += x[k];
  if (s == 12345.678) g_fma_sink = s;   // never true for the arguments used; keeps the chains live
}

cudaError_t fp64_fma_rate(double *flops_per_s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  const int blocks = sms * 8, threads = 256;
  float best = 0.f;
  for (int rep = 0; e == cudaSuccess && rep < 4; ++rep) {   // first run warms up; best of the other three
    cudaEventRecord(e0, 0);
    fp64_fma_kernel<<<blocks, threads>>>(0.999999, 1e-7);
    cudaEventRecord(e1, 0);
    e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaGetLastError();
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e == cudaSuccess && rep > 0 && (best == 0.f || ms < best)) best = ms;
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (e != cudaSuccess) return e;
  *flops_per_s = 2.0 * (double)blocks * threads * kFmaChains * kFmaIters / (best * 1e-3);
  return cudaSuccess;
}

// ---------------------------------------------------------------------------------------------------------
// Static scratch of molc_sweep_static_scratch: the per-sweep workspace (moment accumulators, FP32 cell table)
// in an array fixed at build time, reserved when the module is loaded on a device, so that entry point
// allocates nothing.  The host name g_static_scratch is not a device address: its address on a device comes
// from cudaGetSymbolAddress with that device current, looked up once per device and cached.
// ---------------------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

cudaError_t static_scratch_address(void **ptr) {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static void *cached[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  if (dev >= 0 && dev < kMaxDevices && cached[dev]) {
    *ptr = cached[dev];
    return cudaSuccess;
  }
  void *addr = nullptr;
  e = cudaGetSymbolAddress(&addr, g_static_scratch);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < kMaxDevices) cached[dev] = addr;
  *ptr = addr;
  return cudaSuccess;
}


// =========================================================================================================
// Tiled FP32 sweep: the characteristic grid cut into per-tile pieces (molc_tiles.cpp), one persistent launch
// over work items (tile, quadrant, group tile) taken from an atomic ticket in wavefront order.  Per item:
//   1. one thread starts bulk copies (cp.async.bulk, completion on an mbarrier) of the item's previous-step state
//      (its pieces' deviations, packed step by step exactly as the item walks them) and of its cell table into
//      shared memory, and waits (bounded) until the items upstream in its quadrant have finished this step;
//   2. each thread walks one (piece, group): the deviation-form update of Eqs. 11-13, arithmetic identical to
//      sweep_fp32_body, with the state read and rewritten in shared memory and the records (cell, l) prefetched
//      four steps ahead from L2; the intensity leaving the tile goes to the next piece's slot of the boundary
//      buffer (L2), the item's flag is raised, and the new state is bulk-copied back;
//   3. each thread sums one cell's moment entries of this quadrant from the new state in shared memory (polar
//      fold in FP32, runs of one pair in FP32, two-word FP32 across runs) and writes the quadrant's partial
//      moments (FP64); the last of the four quadrant items of a (tile, group tile) adds the four partials in
//      quadrant order and assembles E, F, N (and f) like the moment gather.
// No block waits on a block that has not started: a ticket is taken only by a running block, and an item waits
// only on items of earlier tickets.  Every wait is bounded and records kStatusTimeout when it gives up.
// =========================================================================================================
namespace {

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// global -> shared bulk copy (16-byte aligned addresses, size a multiple of 16), completing on `bar`
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// shared -> global bulk copy in the issuing thread's bulk group
__device__ __forceinline__ void bulk_store(void *dst, const void *src, unsigned bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// order this thread's shared-memory writes before later bulk copies (async proxy) read them
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ int ld_acquire_gpu(const int *p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(int *p, int v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

constexpr unsigned kBulkChunk = 32768;   // bytes per bulk-copy instruction

// shared memory of one block: state | cdat (float4) | cdB | P | direction table | split-cell partials (double)
struct TileSmem {
  size_t state, cdat, cdB, P, dir, split, total;
};
__host__ __device__ inline size_t up16(size_t b) { return (b + 15) / 16 * 16; }
__host__ __device__ inline TileSmem tile_smem_layout(int max_item_floats, int TS2p, int GT, int max_len,
                                                     int n_pairs, int np, int split_units) {
  TileSmem m;
  m.state = 0;
  m.cdat = up16((size_t)max_item_floats * 4);
  m.cdB = m.cdat + (size_t)GT * TS2p * 16;
  m.P = m.cdB + up16((size_t)GT * TS2p * 4);
  m.dir = m.P + up16((size_t)(max_len + 1) * 4);
  m.split = m.dir + up16((size_t)n_pairs * (3 * np + 2) * 4);
  m.total = m.split + (size_t)split_units * GT * kOutputs * 8;
  return m;
}

// Bounded spin of one thread on a flag reaching `epoch`; false (and the status recorded) if it gave up.  Once a
// wait of the plan has given up, later ones do not wait at all (the step's results are void anyway).
__device__ bool wait_flag(const int *flag, int epoch, int *status) {
  for (int it = 0; it < kTileWaitLimit; ++it) {
    if (ld_acquire_gpu(flag) >= epoch) return true;
    if ((it & 255) == 255 && (*(volatile int *)status & kStatusTimeout)) return false;
    __nanosleep(it < 64 ? 32 : 256);
  }
  atomicOr(status, kStatusTimeout);
  return false;
}

// Cell tables of the tiles (prep_tiles, laid out [tile][G][TS2p], the state's rescale folded into the second
// entry), the input checks, the ticket reset of the coming sweep launch and the plan's step epoch.
__device__ __forceinline__ void tile_prep_body(const PlanView &v, const TileView &t, const SweepArgs &a, int4 m,
                                               int *ticket) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;
  if (m.w && threadIdx.x == 0) t.ctrl[1] += 1;   // a new step of this plan: flags of earlier steps are stale
  const int TS = t.TS, TS2 = TS * TS;
  const int tpb = max(1, (int)blockDim.x / TS2);
  const int tile = m.y + threadIdx.x / TS2, cl = threadIdx.x % TS2;
  const int g = m.z;
  bool bad = false, range = false;
  if (threadIdx.x < tpb * TS2 && tile < t.n_tiles) {
    const int ix = (tile % t.ntx) * TS + cl % TS, iy = (tile / t.ntx) * TS + cl / TS;
    if (ix < v.nx && iy < v.ny) {
      const float inv_cdt_f = (float)a.inv_cdt;
      const double sc = a.scale[0];
      const float rescale = (float)a.scale[3];
      const int64_t idx = (int64_t)g * v.ncell + (int64_t)iy * v.nx + ix;
      const double kap = a.kappa[idx], B = a.B[idx];
      bad = bad_input(kap) | bad_input(B);
      const float kt = (float)(kap + a.inv_cdt);
      const float r = __fdiv_rn(inv_cdt_f, kt);
      const double Bs = B * sc;
      range = __double_as_longlong(Bs) >= __double_as_longlong(kScaledMax);
      const float bhi = (float)Bs;
      const float blo = (float)(Bs - f32_to_f64_exact(bhi));
      const int64_t o = ((int64_t)tile * v.G + g) * t.TS2p + cl;
      t.cdat[o] = make_float4(kt, r * rescale, bhi, blo);
      t.cdB[o] = (float)((a.Bref[idx] - B) * sc) * r;
    }
  }
  if (m.w)
    for (int i = threadIdx.x; i < 4 * v.G; i += blockDim.x) {
      bad |= bad_input(a.bnd[i]);
      range |= !(a.bnd[i] * a.scale[0] < kScaledMax);
    }
  if (bad) atomicOr(v.status, kStatusNonfinite);
  if (range && !bad) atomicOr(v.status, kStatusRange);
}

// map[block] = {instance, first tile, group, 1: this block also checks the boundary and starts the plan's step}
__global__ void __launch_bounds__(256) tile_prep_kernel(const TileInst *inst, const int4 *map, int *ticket) {
  const int4 m = map[blockIdx.x];
  const TileInst &I = inst[m.x];
  tile_prep_body(I.v, I.t, I.a, m, ticket);
}

// One plan: the call's instance comes by value and is stored for the sweep launch that follows.
__global__ void __launch_bounds__(256) tile_prep_one_kernel(TileInst ov, TileInst *dst, const int4 *map,
                                                            int *ticket) {
  const int4 m = map[blockIdx.x];
  if (blockIdx.x == 0 && threadIdx.x == 0) *dst = ov;
  tile_prep_body(ov.v, ov.t, ov.a, m, ticket);
}

// Moments of one cell unit (entries [e0, e1) of the geometry) from the new state in shared memory: polar fold
// in FP32, runs of at most kPairRun entries of one pair in FP32, two-word FP32 across runs (as the moment
// gather), then FP64.
template <int NPM, bool EXACT>
__device__ __forceinline__ void tile_unit_sums(const TileView &t, const TileGeom &gm, int np, int gcnt, int gl,
                                               const float *sst, const float *dirt, int e0, int e1,
                                               double (&D)[kOutputs]) {
  float hi[kOutputs], lo[kOutputs];
#pragma unroll
  for (int k = 0; k < kOutputs; ++k) hi[k] = lo[k] = 0.f;
  const int dstride = 3 * np + 2;
  int cur = -1, run = 0;
  float P0 = 0.f, P1 = 0.f, P2 = 0.f;
  auto flush = [&]() {
    if (cur < 0) return;
    const float cf = dirt[cur * dstride + 3 * np], sf = dirt[cur * dstride + 3 * np + 1];
    two_sum_add(hi[0], lo[0], P0);
    two_sum_add(hi[1], lo[1], cf * P1);
    two_sum_add(hi[2], lo[2], sf * P1);
    two_sum_add(hi[3], lo[3], (cf * cf) * P2);
    two_sum_add(hi[4], lo[4], (cf * sf) * P2);
    two_sum_add(hi[5], lo[5], (sf * sf) * P2);
  };
  const int2 *ent = t.ents + gm.ent_off;
  constexpr int kBatch = 8;   // entries loaded together (their L2 latencies overlap)
  for (int eb = e0; eb < e1; eb += kBatch) {
    int2 enb[kBatch];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) enb[b] = eb + b < e1 ? __ldg(ent + eb + b) : make_int2(0, 0);
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      if (eb + b >= e1) break;
      const int2 en = enb[b];
      const int slot = en.x & 0xFFFFFF, pr = (int)((unsigned)en.x >> 24);
      if (pr != cur || run == kPairRun) {
        flush();
        cur = pr;
        run = 0;
        P0 = P1 = P2 = 0.f;
      }
      ++run;
      const float *dv = sst + ((int64_t)slot * gcnt + gl) * np;
      const float *c0 = dirt + pr * dstride;
      float S0 = 0.f, S1 = 0.f, S2 = 0.f;
#pragma unroll
      for (int p = 0; p < NPM; ++p)
        if (EXACT || p < np) {
          const float x = dv[p];
          S0 = fmaf(c0[p], x, S0);
          S1 = fmaf(c0[np + p], x, S1);
          S2 = fmaf(c0[2 * np + p], x, S2);
        }
      const float af = __int_as_float(en.y);
      P0 = fmaf(af, S0, P0);
      P1 = fmaf(af, S1, P1);
      P2 = fmaf(af, S2, P2);
    }
  }
  flush();
#pragma unroll
  for (int k = 0; k < kOutputs; ++k) D[k] = f32_to_f64(hi[k]) + f32_to_f64(lo[k]);
}

template <int NPM, bool EXACT>
__global__ void __launch_bounds__(512) tile_sweep_kernel(const TileInst *inst, const int2 *queue, int n_queue,
                                                        int *ticket, TileSmem lay) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ unsigned long long bar;
  __shared__ int s_q, s_last;
  float *sst = reinterpret_cast<float *>(smem + lay.state);
  float4 *scd = reinterpret_cast<float4 *>(smem + lay.cdat);
  float *scdB = reinterpret_cast<float *>(smem + lay.cdB);
  int *sP = reinterpret_cast<int *>(smem + lay.P);
  float *sdir = reinterpret_cast<float *>(smem + lay.dir);
  double *ssplit = reinterpret_cast<double *>(smem + lay.split);
  const int tid = threadIdx.x, nthr = blockDim.x;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_proxy_async_smem();
  }
  __syncthreads();
  unsigned phase = 0;
  bool stored = false;   // a bulk store of this block may still be reading shared memory
  int next_q = 0;        // thread 0: the ticket taken for the next item while this one runs
  if (tid == 0) next_q = atomicAdd(ticket, 1);
  for (;;) {
    if (tid == 0) s_q = next_q;
    __syncthreads();
    const int qi = s_q;
    if (qi >= n_queue) break;
    // Take the next ticket now (its latency overlaps this item).  Still no block waits on one that has not
    // started: the smallest unfinished ticket is either some block's current item (its upstream items hold
    // smaller tickets, all finished) or a block's next item whose current item, smaller still, is unfinished.
    if (tid == 0) next_q = atomicAdd(ticket, 1);
    const int2 qe = queue[qi];
    const TileInst &I = inst[qe.x];
    const PlanView &v = I.v;
    const TileView &t = I.t;
    const SweepArgs &a = I.a;
    const int item = qe.y;
    const int gt = item / t.n_geoms, gidx = item - gt * t.n_geoms;
    const TileGeom gm = t.geoms[gidx];
    const int np = EXACT ? NPM : v.n_polar;
    const int g0 = gt * t.GT, gcnt = min(t.GT, v.G - g0);
    const int epoch = t.ctrl[1];
    float *state_g = (float *)a.I + t.item_off[item];
    const unsigned state_bytes = (unsigned)((((int64_t)gm.n_slots * gcnt * np + 3) / 4 * 4) * 4);
    const int64_t cd_off = ((int64_t)gm.tile * v.G + g0) * t.TS2p;
    // 1. stage the state and the cell table (one thread), wait for the upstream items (one thread)
    if (tid == 0) {
      if (stored) bulk_wait_read_all();   // the previous item's store has read the buffer
      const unsigned cd_bytes = (unsigned)gcnt * t.TS2p * 16, cdB_bytes = (unsigned)gcnt * t.TS2p * 4;
      mbar_arrive_expect_tx(&bar, state_bytes + cd_bytes + cdB_bytes);
      for (unsigned o = 0; o < state_bytes; o += kBulkChunk)
        bulk_load((char *)sst + o, (const char *)state_g + o, min(kBulkChunk, state_bytes - o), &bar);
      bulk_load(scd, t.cdat + cd_off, cd_bytes, &bar);
      bulk_load(scdB, t.cdB + cd_off, cdB_bytes, &bar);
    }
    for (int i = tid; i <= gm.max_len; i += nthr) sP[i] = t.Ptab[gm.P_off + i];
    {
      // direction table of this quadrant: per pair the polar folds {w, w sin, w sin^2} and the in-plane
      // direction of the pair's sense that points into q
      const int dstride = 3 * np + 2;
      for (int i = tid; i < v.n_pairs * dstride; i += nthr) {
        const int pr = i / dstride, k = i - pr * dstride;
        float val;
        if (k < 3 * np) {
          const int p = k % np, kind = k / np;
          const PolarDev pd = v.polar[pr * np + p];
          val = kind == 0 ? pd.wf : kind == 1 ? pd.wf * pd.sinzf : (pd.wf * pd.sinzf) * pd.sinzf;
        } else {
          const PairDev pp = v.pairs[pr];
          const bool minus = ((pp.c < 0) != ((gm.q & 1) != 0)) || ((pp.s < 0) != ((gm.q & 2) != 0));
          const float cf = minus ? -pp.cf : pp.cf, sf = minus ? -pp.sf : pp.sf;
          val = k == 3 * np ? cf : sf;
        }
        sdir[i] = val;
      }
    }
    if (tid == 0) {
      const int base = gt * t.n_geoms;
      if (gm.up_x >= 0) wait_flag(t.flags + base + gm.up_x, epoch, v.status);
      if (gm.up_y >= 0) wait_flag(t.flags + base + gm.up_y, epoch, v.status);
      int it = 0;
      while (!mbar_try_wait(&bar, phase) && ++it < kTileWaitLimit) {
        if ((it & 255) == 0 && (*(volatile int *)v.status & kStatusTimeout)) break;   // the step is void already
        __nanosleep(32);
      }
      if (it >= kTileWaitLimit) atomicOr(v.status, kStatusTimeout);
    }
    __syncthreads();
    // all threads observe the completed phase (the copies' data is visible to them after this wait)
    {
      int it = 0;
      while (!mbar_try_wait(&bar, phase) && ++it < kTileWaitLimit) {
        if ((it & 255) == 0 && (*(volatile int *)v.status & kStatusTimeout)) break;
        __nanosleep(32);
      }
    }
    phase ^= 1;
    // 2. walk the pieces
    const double sc = a.scale[0];
    for (int k = tid; k < gm.n_pieces * gcnt; k += nthr) {
      const int r = k / gcnt, gl = k - r * gcnt, g = g0 + gl;
      const int4 pc = t.pieces[gm.piece_off + r];
      const int len = pc.y >> 1;
      const int pair = v.tracks[pc.x].pair;
      float half_inv_sinz[NPM], sinz[NPM], psi[NPM];
#pragma unroll
      for (int p = 0; p < NPM; ++p) {
        half_inv_sinz[p] = sinz[p] = psi[p] = 0.f;
        if (EXACT || p < np) {
          const PolarDev pd = v.polar[pair * np + p];
          half_inv_sinz[p] = 0.5f * pd.inv_sinzf;
          sinz[p] = pd.sinzf;
        }
      }
      float bhi_prev, blo_prev;
      if (pc.z < 0) {   // the piece starts on the domain boundary: entering intensity, split like B
        const double bin = a.bnd[(-1 - pc.z) * v.G + g] * sc;
        bhi_prev = (float)bin;
        blo_prev = (float)(bin - (double)bhi_prev);
      } else {          // from the previous piece of the characteristic (through L2)
        const float *bb = t.bbuf + ((int64_t)pc.z * v.G + g) * (np + 2);
#pragma unroll
        for (int p = 0; p < NPM; ++p)
          if (EXACT || p < np) psi[p] = __ldcg(bb + p);
        bhi_prev = __ldcg(bb + np);
        blo_prev = __ldcg(bb + np + 1);
      }
      const int2 *rec = t.recs + gm.slot_base + r;
      int2 rr[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) rr[u] = u < len ? ld_record(rec + sP[u]) : make_int2(0, 0);
      for (int s0 = 0; s0 < len; s0 += 4) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int s = s0 + u;
          if (s < len) {
            const int2 rc = rr[u];
            if (s + 4 < len) rr[u] = ld_record(rec + sP[s + 4]);
            float *sv = sst + ((int64_t)(sP[s] + r) * gcnt + gl) * np;
            const float4 q = scd[gl * t.TS2p + rc.x];
            const float dB = scdB[gl * t.TS2p + rc.x];
            const float len_f = __int_as_float(rc.y);
            const float jump = (bhi_prev - q.z) + (blo_prev - q.w);
            const float kl = q.x * len_f;
            const float rkl = rcp_approx(kl);
            float dv[NPM];
            if constexpr (NPM == 4) {
              if (EXACT) {
                const float4 d4 = *reinterpret_cast<const float4 *>(sv);
                dv[0] = d4.x;
                dv[1] = d4.y;
                dv[2] = d4.z;
                dv[3] = d4.w;
              } else {
#pragma unroll
                for (int p = 0; p < NPM; ++p) dv[p] = p < np ? sv[p] : 0.f;
              }
            } else {
#pragma unroll
              for (int p = 0; p < NPM; ++p) dv[p] = (EXACT || p < np) ? sv[p] : 0.f;
            }
#pragma unroll
            for (int p = 0; p < NPM; ++p) psi[p] += jump;
#pragma unroll
            for (int p = 0; p < NPM; ++p) {
              if (EXACT || p < np) {
                float E1, om, ex;
                bool thin;
                const float ahalf = kl * half_inv_sinz[p];
                attenuation(ahalf, sinz[p] * rkl, E1, om, ex, thin);
                const float d = fmaf(dv[p], q.y, dB);
                const float pin = psi[p];
                const float x = pin - d;
                dv[p] = fmaf(x, E1, d);
                psi[p] = thin ? fmaf(-x, om, pin) : fmaf(x, ex, d);
              }
            }
            if constexpr (NPM == 4) {
              if (EXACT) {
                *reinterpret_cast<float4 *>(sv) = make_float4(dv[0], dv[1], dv[2], dv[3]);
              } else {
#pragma unroll
                for (int p = 0; p < NPM; ++p)
                  if (p < np) sv[p] = dv[p];
              }
            } else {
#pragma unroll
              for (int p = 0; p < NPM; ++p)
                if (EXACT || p < np) sv[p] = dv[p];
            }
            bhi_prev = q.z;
            blo_prev = q.w;
          }
        }
      }
      if (pc.w >= 0) {   // hand the outgoing intensity to the next piece
        float *bb = t.bbuf + ((int64_t)pc.w * v.G + g) * (np + 2);
#pragma unroll
        for (int p = 0; p < NPM; ++p)
          if (EXACT || p < np) __stcg(bb + p, psi[p]);
        __stcg(bb + np, bhi_prev);
        __stcg(bb + np + 1, blo_prev);
      }
    }
    fence_proxy_async_smem();   // this thread's state writes before the bulk store reads them
    __syncthreads();
    if (tid == 0) {
      if (state_bytes) {
        for (unsigned o = 0; o < state_bytes; o += kBulkChunk)
          bulk_store((char *)state_g + o, (const char *)sst + o, min(kBulkChunk, state_bytes - o));
        bulk_commit();
        stored = true;
      }
      __threadfence();   // every thread's boundary writes (ordered by the barrier) before the flag
      st_release_gpu(t.flags + item, epoch);
    }
    // 3. moments of this quadrant: split cells' parts into shared memory first, then one task per (cell, group)
    const int TS2 = t.TS * t.TS;
    const int2 *cu = t.cell_units + gm.cu_off;
    const int4 *un = t.units + gm.unit_off;
    if (lay.total > lay.split) {
      for (int k = tid; k < gm.n_units * gcnt; k += nthr) {
        const int u = k / gcnt, gl = k - u * gcnt;
        const int4 uu = un[u];
        if (cu[uu.x].y > 1) {
          double D[kOutputs];
          tile_unit_sums<NPM, EXACT>(t, gm, np, gcnt, gl, sst, sdir, uu.y, uu.z, D);
#pragma unroll
          for (int o = 0; o < kOutputs; ++o) ssplit[((int64_t)u * gcnt + gl) * kOutputs + o] = D[o];
        }
      }
      __syncthreads();
    }
    double *part = t.part + (((int64_t)gm.tile * t.n_gt + gt) * 4 + gm.q) * kOutputs * t.GT * t.TS2p;
    for (int k = tid; k < TS2 * gcnt; k += nthr) {
      const int gl = k / TS2, cl = k - gl * TS2;
      const int2 c = cu[cl];
      double D[kOutputs] = {0, 0, 0, 0, 0, 0};
      if (c.y == 1) {
        const int4 uu = un[c.x];
        tile_unit_sums<NPM, EXACT>(t, gm, np, gcnt, gl, sst, sdir, uu.y, uu.z, D);
      } else {
        for (int j = 0; j < c.y; ++j)
#pragma unroll
          for (int o = 0; o < kOutputs; ++o) D[o] += ssplit[((int64_t)(c.x + j) * gcnt + gl) * kOutputs + o];
      }
#pragma unroll
      for (int o = 0; o < kOutputs; ++o) part[((int64_t)o * t.GT + gl) * t.TS2p + cl] = D[o];
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      int *cnt = t.cnt + (int64_t)gm.tile * t.n_gt + gt;
      const int prev = atomicAdd(cnt, 1);
      s_last = prev == 3;
      if (prev == 3) {
        *cnt = 0;   // ready for the next step (its items start after this launch ends)
        __threadfence();
      }
    }
    __syncthreads();
    if (s_last) {   // the four quadrant partials are in place: assemble the tile's cells
      const double *pt = t.part + ((int64_t)gm.tile * t.n_gt + gt) * 4 * kOutputs * t.GT * t.TS2p;
      const int tx = gm.tile % t.ntx, ty = gm.tile / t.ntx;
      for (int k = tid; k < TS2 * gcnt; k += nthr) {
        const int gl = k / TS2, cl = k - gl * TS2;
        const int ix = tx * t.TS + cl % t.TS, iy = ty * t.TS + cl / t.TS;
        if (ix >= v.nx || iy >= v.ny) continue;
        double D[kOutputs] = {0, 0, 0, 0, 0, 0};
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int o = 0; o < kOutputs; ++o)
            D[o] += __ldcg(pt + (((int64_t)q * kOutputs + o) * t.GT + gl) * t.TS2p + cl);
        assemble_cell(v, a, iy * v.nx + ix, g0 + gl, D);
      }
    }
    __syncthreads();
  }
  if (tid == 0 && stored) bulk_wait_all();   // the last state store has completed
}

// Canonical segment averages <-> tiled FP32 state: one thread per row (track, sense, step), looping over polar
// cosines and the selected groups (as intensity_copy_kernel; only the element address differs).
__global__ void tile_intensity_copy_kernel(PlanView v, TileView t, const int4 *tpiece, const int64_t *tpiece_off,
                                           float *I, const double *Bref, const double *scale, int g_begin,
                                           int g_count, double *canon, int to_canon, int64_t rows) {
  const int NP = v.n_polar;
  const double sc = scale[0], is = scale[1];
  for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < rows;
       row += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = find_track(v.tracks, v.n_tracks, row);
    const TrackDev tr = v.tracks[k];
    const int64_t local = row - 2 * tr.seg_off;
    const int sense = local >= tr.nseg;
    const int s = (int)(local - (int64_t)sense * tr.nseg);
    const int cell = v.seg_cell[sense ? tr.seg_off + tr.nseg - 1 - s : tr.seg_off + s];
    // the piece holding step s of this sense
    const int64_t a0 = tpiece_off[2 * k + sense], a1 = tpiece_off[2 * k + sense + 1];
    int64_t pi = a0;
    while (pi + 1 < a1 && tpiece[pi + 1].z <= s) ++pi;
    const int4 tp = tpiece[pi];
    const TileGeom gm = t.geoms[tp.x];
    const int slot = t.Ptab[gm.P_off + (s - tp.z)] + tp.y;
    for (int p = 0; p < NP; ++p) {
      const PolarDev pd = v.polar[tr.pair * NP + p];
      const int dir = sense ? pd.dir_minus : pd.dir_plus;
      const int64_t cs = v.dir_seg_off[dir] + (sense ? tr.canon_minus : tr.canon_plus) + s;
      for (int g = g_begin; g < g_begin + g_count; ++g) {
        const int gt = g / t.GT, gl = g - gt * t.GT, gcnt = min(t.GT, v.G - gt * t.GT);
        float *el = I + t.item_off[(int64_t)gt * t.n_geoms + tp.x] + ((int64_t)slot * gcnt + gl) * NP + p;
        const double br = Bref[(int64_t)g * v.ncell + cell];
        double *cv = canon + cs * g_count + (g - g_begin);
        if (to_canon)
          *cv = br + (double)*el * is;
        else
          *el = (float)((*cv - br) * sc);
      }
    }
  }
}

// Allow a kernel the device's largest dynamic shared memory (the opt-in limit less its static shared memory).
cudaError_t allow_max_dynamic_smem(const void *fn) {
  int dev = 0, optin = 0;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, fn);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
  if (e != cudaSuccess) cudaGetLastError();   // do not leave the error for a later launch check
  return e;
}

template <int NPM, bool EXACT>
cudaError_t launch_tile_np(const TileInst *inst, const int2 *queue, int n_queue, int *ticket, const TileSmem &lay,
                           int grid, int threads, cudaStream_t st) {
  static bool attr = false;   // once per instantiation
  if (!attr) {
    cudaError_t e = allow_max_dynamic_smem((const void *)tile_sweep_kernel<NPM, EXACT>);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  tile_sweep_kernel<NPM, EXACT><<<grid, threads, lay.total, st>>>(inst, queue, n_queue, ticket, lay);
  return cudaGetLastError();
}

}  // namespace

size_t tile_sweep_smem(const TileShape &sh, int np_max) {
  return tile_smem_layout(sh.max_item_floats, sh.cd_entries, 1, sh.max_len, sh.n_pairs, np_max, sh.split_units).total;
}

cudaError_t launch_tile_prep(const TileInst *inst, const int4 *map, int blocks, int *ticket, cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  tile_prep_kernel<<<blocks, 256, 0, st>>>(inst, map, ticket);
  return cudaGetLastError();
}

cudaError_t launch_tile_prep_one(const TileInst &ov, TileInst *dst, const int4 *map, int blocks, int *ticket,
                                 cudaStream_t st) {
  if (blocks <= 0) return cudaSuccess;
  tile_prep_one_kernel<<<blocks, 256, 0, st>>>(ov, dst, map, ticket);
  return cudaGetLastError();
}

cudaError_t launch_tile_sweep(const TileInst *inst, const int2 *queue, int n_queue, int *ticket, int np_max,
                              const TileShape &sh, int grid, int threads, cudaStream_t st) {
  const TileSmem lay = tile_smem_layout(sh.max_item_floats, sh.cd_entries, 1, sh.max_len, sh.n_pairs, np_max,
                                        sh.split_units);
  const bool exact = sh.np_exact == np_max;
  switch (np_max) {
    case 1: return exact ? launch_tile_np<1, true>(inst, queue, n_queue, ticket, lay, grid, threads, st)
                         : launch_tile_np<1, false>(inst, queue, n_queue, ticket, lay, grid, threads, st);
    case 2: return exact ? launch_tile_np<2, true>(inst, queue, n_queue, ticket, lay, grid, threads, st)
                         : launch_tile_np<2, false>(inst, queue, n_queue, ticket, lay, grid, threads, st);
    case 3: case 4: return exact && np_max == 4 ? launch_tile_np<4, true>(inst, queue, n_queue, ticket, lay, grid, threads, st)
                                                : launch_tile_np<4, false>(inst, queue, n_queue, ticket, lay, grid, threads, st);
    default: return exact && np_max == 8 ? launch_tile_np<8, true>(inst, queue, n_queue, ticket, lay, grid, threads, st)
                                         : launch_tile_np<8, false>(inst, queue, n_queue, ticket, lay, grid, threads, st);
  }
}

int tile_sweep_grid(int np_max, size_t smem, int threads) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const void *fn = np_max <= 1 ? (const void *)tile_sweep_kernel<1, true>
                 : np_max <= 2 ? (const void *)tile_sweep_kernel<2, true>
                 : np_max <= 4 ? (const void *)tile_sweep_kernel<4, true> : (const void *)tile_sweep_kernel<8, true>;
  allow_max_dynamic_smem(fn);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem) != cudaSuccess || per < 1) {
    cudaGetLastError();
    per = 1;
  }
  return sms * per;
}

cudaError_t launch_tile_intensity_copy(const PlanView &v, const TileView &t, const int4 *tpiece,
                                       const int64_t *tpiece_off, float *I, const double *Bref,
                                       const double *scale, int g_begin, int g_count, double *canon, bool to_canon,
                                       cudaStream_t st) {
  const int64_t rows = 2 * v.n_track_segments;
  tile_intensity_copy_kernel<<<grid_for(rows, 128), 128, 0, st>>>(v, t, tpiece, tpiece_off, I, Bref, scale, g_begin,
                                                                  g_count, canon, to_canon, rows);
  return cudaGetLastError();
}

}  // namespace molc
