// Resident step kernel: many steps of one grid in one cooperative launch.
//
// A step alone takes two launches (the streaming step kernel, then the
// finalize kernel); on grids of up to some tens of MB their prologues, the
// launch gaps and the finalize's chain of small dependent reads take longer
// than the update itself.  Here every work unit (fk_stream_unit.cuh) keeps
// its CTA through all the steps, and a few more CTAs of the same launch do
// the finalize: a step is the units' march, one count per unit, the
// finalize, and one "go" that the units wait for.
//
//  - Units: CTA b < n_units runs unit b (tile b % n_tiles, chunk b / n_tiles)
//    with its set-up (tables, cell offsets, mbarriers) done once.
//  - Finalize CTAs: one per 128 planes, as the finalize kernel's blocks, one
//    thread per plane.  They hold the run's scalars and the parameters in
//    shared memory and registers.  Between the units' last arrival and "go"
//    stand only: the planes' partial sums, one scan, one exchange of the
//    block totals (through L2, each value its own flag), E_x and c_1.  The
//    ledger, the history row, the convergence test and the velocity-edge
//    loss follow while the units march on.
// Every sum has the order of finalize_body, so a step is bit for bit the
// one that the two kernels give.
//
// What bounds it: on small grids the chain arrival -> partial sums -> scan ->
// E_x -> go (about 3.5 us on one finalize CTA, 5 us on several) and the unit
// that holds the wall; on large ones HBM (FP32) or the FP64 pipe.  Measured, us
// a step, two launches a step replayed as graphs -> here: 64 x 48 x 48 FP64 34.9
// -> 15.4, FP32 20.4 -> 10.4; 321 x 117 x 117 FP32 26.2 -> 21.6; 512 x 128 x 128
// FP32 with collisions and reflection 33.0 -> 26.2; 1024 x 256 x 256 FP32 109.7
// -> 105.3, FP64 620 -> 576.  (The FP32 kernels of whole-CTA units spill 52 to
// 116 bytes; the two-launch step kernel of the largest grid takes 99.7 us of its
// 109.7 without a spill.)
//
// Waits: every block of the launch is resident (cooperative launch), every
// wait is bounded by Params::wait_limit, and after one that runs out the
// launch ends with kFlagTimeout set and the state of the last whole step.  A
// finalize CTA that finds a Courant or non-finite fault in the new state ends
// the launch after that step, through both counters (kGoStop).
#include <stddef.h>

#include <algorithm>

#include "fk_finalize.cuh"
#include "fk_resident.cuh"
#include "fk_stream_unit.cuh"

namespace fk {

namespace {

constexpr int kThinBlock = kHalfThreads + 32;  // a CTA of one thin unit
static_assert(kThinBlock >= kFinThreads && kBlock >= kFinThreads, "a finalize CTA's threads");

// A slot of the block exchange that holds no value yet: a NaN no sum gives
// (a sum that is this very pattern is written as another NaN).
constexpr unsigned long long kNoValue = 0xFFFFFFFFFFFFFFFFull;

__device__ __forceinline__ void fin_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kFinThreads) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void put_value(unsigned long long* p, double x) {
  unsigned long long v = (unsigned long long)__double_as_longlong(x);
  if (v == kNoValue) v = 0x7FF8000000000000ull;
  st_relaxed64(p, v);
}
// The value another block puts into slot p; *ok = false if the wait ran out.
__device__ __forceinline__ double take_value(const unsigned long long* p, long long lim, bool* ok) {
  unsigned long long v = ld_relaxed64(p);
  const long long t0 = clock64();
  while (v == kNoValue) {
    if (clock64() - t0 > lim) {
      *ok = false;
      return 0.0;
    }
    v = ld_relaxed64(p);
  }
  return __longlong_as_double((long long)v);
}

// The exchange's rows of kFinMaxBlocks slots: two for the densities (even and
// odd steps), then three for the velocity-edge sums.
constexpr int kXchRows = 5;
__device__ __forceinline__ unsigned long long* lv_slots(const ResidentArgs& ra, int step) {
  return ra.xch + (size_t)(2 + step % 3) * kFinMaxBlocks;
}

// sum over tiles of plane k's partials, in tile order (as finalize_body)
__device__ __forceinline__ double plane_sum(const double* p, int nu) {
  double s = 0.0;
  int u = 0;
  for (; u + 8 <= nu; u += 8) {
    double x[8];
#pragma unroll
    for (int q = 0; q < 8; q++) x[q] = __ldcg(p + u + q);
#pragma unroll
    for (int q = 0; q < 8; q++) s += x[q];
  }
  for (; u < nu; u++) s += __ldcg(p + u);
  return s;
}

// sum over the warp, lanes >= n holding zeros; valid in lane 0
__device__ __forceinline__ double warp_tree(double v, int n = 32) {
  for (int o = 16; o > 0; o >>= 1)
    if (o < n) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Finalize CTA blk of n_fin: steps 0 .. n_steps - 1 of the launch, with
// kFinThreads threads, plane k = blk * kFinThreads + thread.
struct FinShared {
  double wscan[kFinThreads / 32], lsum[kFinThreads / 32];
  double wall[3];   // Gamma_pe, Gamma_see, Gamma_vac of the new state
  double off, n;    // densities below this block; of all planes
  double sigma;     // sigma of the new state
  // stop: the step's inputs are void, leave before it; end: this block found a
  // fault in the new state, leave after the step.  Two words: end is read after
  // the step's last barrier, when thread 0 may already be setting stop for the
  // next one.
  int stop, end, bad;
  DevState d;       // block 0: the run's scalars
};

__device__ __forceinline__ void resident_finalize(const ResidentArgs& ra, const int blk,
                                                  FinShared& sh) {
  const StepArgs& a = ra.a;
  const FinOut& o = ra.o;
  const Params& p = *a.prm;
  DevState* st = a.st;
  const int n_fin = (int)ra.rs.n_fin;
  const int nx = a.nx, nu = a.part.nu;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int k = blk * kFinThreads + t;
  const bool live = k < nx;
  const double dvv = p.dvv, ex_sigma = p.ex_sigma, ex_n = p.ex_n, ex_ext = p.Ex_ext;
  const double c1_per_ex = p.c1_per_ex, bgk_c = p.bgk_c, cx_max = p.cx_max, ac2 = fabs(p.c2);
  const double refl = p.refl, dt = p.dt;
  const bool self_cons = p.self_consistent, coll = p.collisions, see_on = p.see_enabled;
  const long long lim = p.wait_limit;
  if (t == 0) {
    sh.d = *st;
    sh.sigma = advance_sigma(sh.d.sigma, dt, sh.d.g_see, sh.d.g_pe, refl);
    sh.stop = sh.end = sh.bad = 0;
  }
  fin_sync();
  for (int step = 0; step < ra.rs.n_steps; step++) {
    // ---- every unit has finished the step
    if (t == 0) {
      const unsigned want = ra.rs.n_units * (unsigned)(step + 1);
      const long long t0 = clock64();
      while (read_count(ra.rs.arrive) < want)
        if (clock64() - t0 > lim) {
          atomicOr(&st->flags, kFlagTimeout);
          break;
        }
      if (__ldcg(&st->flags)) sh.stop = 1;
    }
    fin_sync();
    if (sh.stop) {  // the state stays that of the last whole step
      if (t == 0) count_arrival(ra.rs.go, kGoStop);
      return;
    }
    // ---- the planes' densities, their prefix, and the wall fluxes
    double nk = 0.0;
    if (live) nk = plane_sum(a.part.n + (size_t)k * nu, nu) * dvv;
    double incl = nk;
    for (int d = 1; d < 32; d <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += y;
    }
    double excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) excl = 0.0;
    if (lane == 31) sh.wscan[w] = incl;
    if (w == 3) {  // its tree in the shadow of the exchange below
      double pe = 0.0, see = 0.0, vac = 0.0;
      for (int u = lane; u < nu; u += 32) {
        pe += __ldcg(a.part.pe + u);
        see += __ldcg(a.part.see + u);
        vac += __ldcg(a.part.vac + u);
      }
      pe = warp_tree(pe, nu);
      see = warp_tree(see, nu);
      vac = warp_tree(vac, nu);
      if (lane == 0) {
        sh.wall[0] = pe * dvv;
        sh.wall[1] = see_on ? see * dvv * (1.0 - refl) : 0.0;
        sh.wall[2] = vac * dvv;
      }
    }
    fin_sync();
    double woff = 0.0, btot = 0.0;
    for (int q = 0; q < kFinThreads / 32; q++) {
      if (q == w) woff = btot;
      btot += sh.wscan[q];
    }
    const double pre = woff + excl;
    if (n_fin > 1) {  // block totals: all to all
      unsigned long long* slot = ra.xch + (size_t)(step & 1) * kFinMaxBlocks;
      if (w == 0) {
        if (lane == 0) {
          put_value(slot + blk, btot);
          // this block's slots of the next step, emptied before this step's
          // release of go, which orders that before any read in the next one.
          // The last reads of those slots lie before a go that this block has
          // seen the units pass: a step back for the densities, read before it;
          // two for the velocity-edge sums, read after it (a third row).
          st_relaxed64(ra.xch + (size_t)((step + 1) & 1) * kFinMaxBlocks + blk, kNoValue);
          st_relaxed64(lv_slots(ra, step + 1) + blk, kNoValue);
        }
        bool ok = true;
        const double b0 = lane < n_fin ? take_value(slot + lane, lim, &ok) : 0.0;
        const double b1 = lane + 32 < n_fin ? take_value(slot + lane + 32, lim, &ok) : 0.0;
        double i0s = b0, i1s = b1;
        for (int d = 1; d < 32; d <<= 1) {
          if (d >= n_fin) break;
          const double y0 = __shfl_up_sync(0xffffffffu, i0s, d);
          if (lane >= d) i0s += y0;
        }
        if (n_fin > 32)
          for (int d = 1; d < 32; d <<= 1) {
            const double y1 = __shfl_up_sync(0xffffffffu, i1s, d);
            if (lane >= d) i1s += y1;
          }
        const double half = __shfl_sync(0xffffffffu, i0s, min(n_fin, 32) - 1);
        const double total = n_fin > 32 ? half + __shfl_sync(0xffffffffu, i1s, n_fin - 33) : half;
        if (lane == (blk & 31)) {
          sh.off = blk < 32 ? i0s - b0 : half + i1s - b1;
          sh.n = total;
        }
        if (__any_sync(0xffffffffu, !ok) && lane == 0) {
          atomicOr(&st->flags, kFlagTimeout);
          sh.stop = 1;
        }
      }
      fin_sync();
      if (sh.stop) {
        if (t == 0) count_arrival(ra.rs.go, kGoStop);
        return;
      }
    } else if (t == 0) {
      sh.off = btot - btot;  // 0, or NaN as the general form gives
      sh.n = btot;
    }
    if (n_fin == 1) fin_sync();
    // ---- E_x and the coefficients of the next step
    const double below = sh.off + pre;
    const double e_wall = sh.sigma * ex_sigma;
    const double e = self_cons ? field_at(e_wall, ex_n, below, nk) : ex_ext;
    const double c = c1_per_ex * e;
    double ak = 0.0;
    if (live) {
      o.c1[k] = c;
      o.c1_32[k] = (float)c;
      double cfl = fabs(c);
      if (coll) {
        ak = nk > 0.0 ? bgk_c * nk : 0.0;
        a.bgk[k] = ak;
        a.bgk[nx + k] = ak * nk;
        a.bgk32[k] = (float)ak;
        a.bgk32[nx + k] = (float)(ak * nk);
        cfl += ak;
      }
      if (cfl + cx_max + ac2 > 1.0 + 1e-12) sh.bad = 1;
    }
    const double ntot = sh.n * p.dx;
    if (t == 0 && blk == 0) st->g_see = sh.wall[1];
    fin_sync();
    if (t == 0) {
      unsigned bad = sh.bad ? kFlagCfl : 0u;
      if (blk == 0 && (!isfinite(sh.wall[0]) || !isfinite(sh.wall[1]) || !isfinite(sh.wall[2]) ||
                       !isfinite(ntot) || !isfinite(sh.sigma)))
        bad |= kFlagNumeric;
      if (bad) atomicOr(&st->flags, bad);
      // A fault of this block's planes is known to this block alone: the units
      // learn of it through go, the other blocks, which wait for the next
      // step's arrivals, through arrive (every one of them has passed this
      // step's, or the exchange would not have ended).
      if (bad) count_arrival(ra.rs.arrive, kGoStop);
      count_arrival(ra.rs.go, bad ? 1u + kGoStop : 1u);
      sh.end = bad != 0;
    }
    // ---- while the units march on: what only the getters and the ledger read
    if (live) {
      o.ne[k] = nk;
      o.Ex[k] = e;
    }
    double lk = live ? plane_sum((step & 1 ? ra.rs.lv_odd : a.part.lv) + (size_t)k * nu, nu) : 0.0;
    lk = warp_tree(lk);
    if (lane == 0) sh.lsum[w] = lk;
    fin_sync();
    if (w == 0) {
      double l = lane < kFinThreads / 32 ? sh.lsum[lane] : 0.0;
      l = warp_tree(l, kFinThreads / 32);
      bool ok = true;
      if (n_fin > 1) {
        unsigned long long* slot = lv_slots(ra, step);
        if (lane == 0) put_value(slot + blk, l);
        if (blk == 0)
          l = (lane < n_fin ? take_value(slot + lane, lim, &ok) : 0.0) +
              (lane + 32 < n_fin ? take_value(slot + lane + 32, lim, &ok) : 0.0);
      } else {
        l = (lane == 0 ? l : 0.0) + 0.0;
      }
      if (blk == 0) {
        l = warp_tree(l, n_fin);
        if (__any_sync(0xffffffffu, !ok) && lane == 0) atomicOr(&st->flags, kFlagTimeout);
        if (lane == 0) {
          advance_ledger(sh.d, p, l, dt);
          sh.d.sigma = sh.sigma;
          sh.d.g_pe = sh.wall[0];
          sh.d.g_see = sh.wall[1];
          sh.d.g_vac = sh.wall[2];
          sh.d.n_tot = ntot;
          const double ex0 = e;  // thread 0 of block 0 holds plane 0
          append_history(sh.d, p, o.hist, ex0, true);
        }
        __syncwarp();
        // every scalar but the flags, which units may set meanwhile
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&sh.d);
        unsigned long long* dst = reinterpret_cast<unsigned long long*>(st);
        if (lane < (int)(offsetof(DevState, flags) / 8)) dst[lane] = src[lane];
      }
    }
    if (t == 0) sh.sigma = advance_sigma(sh.sigma, dt, sh.wall[1], sh.wall[0], refl);
    fin_sync();
    if (sh.end) return;
  }
}

template <typename T, bool PADDED, bool BGK, int NT>
__global__ void __launch_bounds__(NT + 32, NT == kThreads ? 2 : 4)
resident_kernel(const __grid_constant__ ResidentArgs ra) {
  extern __shared__ __align__(128) unsigned char smem[];
  if (blockIdx.x >= ra.rs.n_units) {
    if (threadIdx.x < kFinThreads)
      resident_finalize(ra, (int)(blockIdx.x - ra.rs.n_units), *reinterpret_cast<FinShared*>(smem));
    return;
  }
  const int nt = ra.a.geom.n_tiles;
  stream_unit<T, PADDED, BGK, NT, false, true>(ra.a, blockIdx.x % nt, blockIdx.x / nt, smem,
                                               threadIdx.x, 0, ra.rs);
}

template <typename T, bool PADDED, bool BGK, int NT>
cudaError_t launch_one(ResidentArgs& ra, int ctas, size_t smem, cudaStream_t s) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(NT + 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, resident_kernel<T, PADDED, BGK, NT>, ra);
}
template <typename T, int NT>
cudaError_t launch_sized(ResidentArgs& ra, int ctas, size_t smem, bool bgk, cudaStream_t s) {
  const bool padded = ra.a.pitch != ra.a.nv2;
  if (padded)
    return bgk ? launch_one<T, true, true, NT>(ra, ctas, smem, s)
               : launch_one<T, true, false, NT>(ra, ctas, smem, s);
  return bgk ? launch_one<T, false, true, NT>(ra, ctas, smem, s)
             : launch_one<T, false, false, NT>(ra, ctas, smem, s);
}

template <typename T, bool PADDED, bool BGK, int NT>
cudaError_t fit_one(int optin, size_t smem, int* best) {
  int n = 0;
  auto kernel = resident_kernel<T, PADDED, BGK, NT>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, NT + 32, smem);
  if (e == cudaSuccess && n < *best) *best = n;
  return e;
}
// the smaller of the variants with and without the collision term, which a
// setter may switch on later
template <typename T, int NT>
int fit_sized(int optin, size_t smem, bool padded) {
  int best = 1 << 30;
  cudaError_t e = padded ? fit_one<T, true, false, NT>(optin, smem, &best)
                         : fit_one<T, false, false, NT>(optin, smem, &best);
  if (e == cudaSuccess)
    e = padded ? fit_one<T, true, true, NT>(optin, smem, &best)
               : fit_one<T, false, true, NT>(optin, smem, &best);
  return e == cudaSuccess ? best : 0;
}

}  // namespace

// two 32-bit counters, each on its own 128-byte line, then the exchange
constexpr int kXchWord = 64;
int resident_scratch_words() { return kXchWord + 2 * kXchRows * kFinMaxBlocks; }

size_t resident_smem_bytes(int precision, const Geom& gm, int pitch) {
  // a unit's block without the argument slot of the batched kernels, with
  // four more control words and the items' values
  size_t n = precision == FK_F32
                 ? (gm.half ? unit_smem_bytes<float, kHalfStages>(gm.stage_elems, pitch)
                            : unit_smem_bytes<float, kStages>(gm.stage_elems, pitch))
                 : (gm.half ? unit_smem_bytes<double, kHalfStages>(gm.stage_elems, pitch)
                            : unit_smem_bytes<double, kStages>(gm.stage_elems, pitch));
  n = n - kArgsBytes + 16 + std::max(kStages, kHalfStages) * sizeof(ItemVals);
  return n < sizeof(FinShared) ? sizeof(FinShared) : n;
}

int resident_ctas_per_sm(int precision, const Geom& gm, int pitch, bool padded) {
  int dev = 0, optin = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
    return 0;
  const size_t smem = resident_smem_bytes(precision, gm, pitch);
  if (smem > (size_t)optin) return 0;
  if (precision == FK_F32)
    return gm.half ? fit_sized<float, kHalfThreads>(optin, smem, padded)
                   : fit_sized<float, kThreads>(optin, smem, padded);
  return gm.half ? fit_sized<double, kHalfThreads>(optin, smem, padded)
                 : fit_sized<double, kThreads>(optin, smem, padded);
}

cudaError_t launch_resident(const StepArgs& a, const FinOut& o, int precision, bool bgk,
                            int n_steps, double* lv_odd, unsigned* scratch, cudaStream_t s) {
  ResidentArgs ra{};
  ra.a = a;
  ra.o = o;
  ra.xch = reinterpret_cast<unsigned long long*>(scratch + kXchWord);
  ra.rs = Resident{scratch, scratch + 32, (unsigned)(a.geom.n_tiles * a.geom.n_chunks),
                   (unsigned)((a.nx + kFinThreads - 1) / kFinThreads),
                   n_steps, lv_odd};
  const int ctas = (int)(ra.rs.n_units + ra.rs.n_fin);
  const size_t smem = resident_smem_bytes(precision, a.geom, a.pitch);
  cudaError_t e = cudaMemsetAsync(scratch, 0xFF, resident_scratch_words() * sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  if (precision == FK_F32)
    return a.geom.half ? launch_sized<float, kHalfThreads>(ra, ctas, smem, bgk, s)
                       : launch_sized<float, kThreads>(ra, ctas, smem, bgk, s);
  return a.geom.half ? launch_sized<double, kHalfThreads>(ra, ctas, smem, bgk, s)
                     : launch_sized<double, kThreads>(ra, ctas, smem, bgk, s);
}

}  // namespace fk
