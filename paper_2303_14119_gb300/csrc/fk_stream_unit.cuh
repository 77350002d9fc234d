// Streaming step kernel: one explicit upwind step of Eq. 2 (Sun et al.,
// arXiv 2303.14119, Sec. 2) over the whole phase-space grid, one read of
// f^n and one write of f^{n+1} per cell.
//
// Decomposition.  A CTA owns one unit = (tile of v1 rows [i0, i1) times all
// v2 cells, chunk of consecutive x-planes), or two units of thin tiles, one
// per half of the CTA.  All rows of a tile have the same sign of v1, so the
// x-upwind neighbour of plane k is plane k - dir for the whole tile; the
// unit marches through its chunk in the direction dir, and every consumer
// thread keeps the previous plane's input values of its own cells in
// registers: the x-neighbour never comes from memory twice.
//
// Pipeline.  Planes arrive in shared memory through cp.async.bulk copies
// (the TMA engine) into a ring of stages (kStages for a whole-CTA unit,
// kHalfStages for a half-CTA unit, whose planes are small).  Each stage holds the
// tile's rows plus the one v1 halo row on the upwind side of that plane's
// c_1.  Warp roles:
//  - consumer warps (kWarps): wait until a stage is full, update their cells
//    (FP32/INT work only on the FP32 path), store f^{n+1}, sum it per warp,
//    and release the stage;
//  - the producer warp: when a stage is released, read what the partial
//    sums of its plane need (the warp sums; the outflow of f^n through the
//    downwind velocity edges, still in the stage), refill the stage, then
//    fold them into the per-(plane, tile) partial sums (on x = 0 and
//    x = h_max with the wall fluxes of Eqs. 12-14 and the vacuum outflow
//    of f^{n+1}).
// There is no block-wide barrier inside the march.
//
// Per cell: f' = f + |c_x|(f_ux - f) + |c_1|(f_u1 - f) + |c_2|(f_u2 - f) + dt S
// (FP32: increment form) or the convex form of the same sum (FP64).
#pragma once

#include <type_traits>
#include <stdint.h>

#include "fk_internal.cuh"
#include "fk_resident.cuh"

namespace fk {
namespace {

constexpr int kThreads = 224;            // consumer threads of a whole-CTA unit (7 warps)
constexpr int kWarps = kThreads / 32;    // its consumer warps; one producer warp follows
constexpr int kBlock = kThreads + 32;
// Thin tiles (few cells per plane) run two units per CTA, each on one half:
// 3 consumer warps and its own producer warp, stages and mbarriers.
constexpr int kHalfThreads = 96;
constexpr int kHalfBlock = kHalfThreads + 32;
static_assert(2 * kHalfBlock == kBlock, "two half units fill one CTA");
constexpr int kStages = 4;      // stages of a whole-CTA unit
constexpr int kHalfStages = 4;  // stages of a half-CTA unit
static_assert(kHalfStages <= 32, "a producer lane per stage");
// stages of a unit on NT consumer threads
template <int NT>
__host__ __device__ constexpr int unit_stages() { return NT == kThreads ? kStages : kHalfStages; }
constexpr int kVecPerThread = 8;         // 16-byte vectors per consumer thread and plane
constexpr int kHalfVecPerThread32 = 3;   // the same for half units of FP32 grids
// vectors per consumer thread and plane of a unit on NT threads, element size E
template <int NT, int E>
__host__ __device__ constexpr int unit_vectors() {
  return (NT == kHalfThreads && E == 4) ? kHalfVecPerThread32 : kVecPerThread;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Order this thread's earlier generic-proxy shared-memory accesses before
// later async-proxy (bulk copy) accesses to the same memory.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for the phase with the given parity; false if it did not complete
// within *limit cycles (read only when the first try fails).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, const long long* limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long lim = *limit;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > lim) return false;
  return true;
}

__device__ __forceinline__ unsigned read_count(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v - kCountZero;
}
// Count one arrival; the caller's unit has synchronised its threads, whose
// writes the fence makes visible before the count.
__device__ __forceinline__ void count_arrival(unsigned* p, unsigned v) {
  __threadfence();
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// This thread's global accesses through one proxy (generic or the bulk
// copies') before later ones through the other.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
// Values other SMs write during the launch are read in L2 (RES), where a
// plain load could find an old copy in this SM's L1.
template <bool RES, typename X>
__device__ __forceinline__ X ld_shared_value(const X* p) {
  if constexpr (RES)
    return __ldcg(p);
  else
    return *p;
}

template <typename T>
struct alignas(16) Vec {
  static constexpr int N = 16 / sizeof(T);
  T e[N];
};

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Two FP32 values in one 64-bit register: each packed operation rounds its two
// results as the scalar operation does, in one instruction instead of two.
using F2 = unsigned long long;
__device__ __forceinline__ F2 f2_pack(float x, float y) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(F2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// a - b: one rounding, as a subtraction
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
  return f2_fma(b, f2_pack(-1.f, -1.f), a);
}

__device__ __forceinline__ double upd(double f, double fx, double fv, double fw, double ax,
                                      double a1, double a2, double s, double d) {
  // every weight is >= 0 under the CFL condition: nothing cancels
  return fma(a2, fw, fma(a1, fv, fma(ax, fx, fma(d, f, s))));
}

template <typename T>
__host__ __device__ constexpr size_t stage_bytes(int stage_elems) {
  return ((size_t)stage_elems * sizeof(T) + 127) / 128 * 128;
}
// The dynamic shared memory of both kernels starts with a slot for the
// unit's StepArgs (filled by the batched kernel), so that one tile plan fits
// a grid stepped alone or in a batch.  After the slot and the stages come:
// mbarriers full[NS], empty[NS] (NS stages); warp sums [NS][kWarps][4]
// (a half unit uses the first 3 warps of each stage)
// (density as one or two floats, wall primary flux, wall secondary flux,
// vacuum outflow); for
// FP64 grids the per-stage diagonal 1 - |c_x| - |c_1| - |c_2| (- dt nu) of
// every tile row [NS][kMaxTileRows] double, for FP32 grids the
// separable source factors of the tile rows [kMaxTileRows] and of the row
// cells [pitch] (float); the BGK equilibrium factors of Eq. 5 (FP32 grids:
// m1 of the tile rows [kMaxTileRows] and m2 [pitch], float; FP64 grids:
// dt nu_k n_k m1 per stage and tile row [NS][kMaxTileRows] and m2
// [pitch], double); control words: the sticky flags and a withheld
// pipeline item (ints), the wait limit (long long, at byte 8).
constexpr int kArgsBytes = 384;  // a multiple of 128: the stages stay 128-byte aligned
static_assert(sizeof(StepArgs) <= kArgsBytes && sizeof(StepArgs) % 8 == 0,
              "StepArgs must fit its shared-memory slot");
constexpr int kWs = 4;
constexpr int kMaxTileRows = 64;  // also bounds the per-stage row tables
template <typename T, int NS>
__host__ __device__ constexpr size_t tail_main_bytes(int pitch) {
  return sizeof(T) == 8 ? NS * kMaxTileRows * sizeof(double)
                        : ((size_t)(kMaxTileRows + pitch) * sizeof(float) + 15) / 16 * 16;
}
template <typename T, int NS>
__host__ __device__ constexpr size_t tail_bgk_bytes(int pitch) {
  return sizeof(T) == 8 ? (NS * kMaxTileRows + (size_t)pitch) * sizeof(double)
                        : ((size_t)(kMaxTileRows + pitch) * sizeof(float) + 15) / 16 * 16;
}
template <typename T, int NS>
__host__ __device__ constexpr size_t tail_bytes(int pitch) {
  return kArgsBytes + 2 * NS * sizeof(uint64_t) + NS * kWarps * kWs * sizeof(double) +
         tail_main_bytes<T, NS>(pitch) + tail_bgk_bytes<T, NS>(pitch) + 16;
}

// Exact split of a double x with 2^-126 <= |x| < 2^128 into hi + lo floats:
// hi keeps the top 24 significant bits (truncated), lo the remaining 29
// rounded to 24 bits, so hi + lo = x to about 2^-47 relative.  Integer and
// FP32 operations only: none of this runs on GB300's narrow FP64 pipe.
// Smaller magnitudes (and zero) give 0 + 0, negligible in a sum of
// phase-space densities; |x| >= 2^128, infinities and NaN give a NaN hi, so
// the sum they enter is flagged as non-finite.
__device__ __forceinline__ void split_double(double x, float& hi, float& lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned int h32 = (unsigned int)(b >> 32);
  const int E = (int)((h32 >> 20) & 0x7FF);
  const unsigned int sign = h32 & 0x80000000u;
  const unsigned int m23 = (unsigned int)(b >> 29) & 0x7FFFFFu;
  const bool ok = E >= 897 && E <= 1150;  // hi is a normal float
  const unsigned int out_of_range = E > 1150 ? 0x7FC00000u : 0u;  // quiet NaN
  hi = __int_as_float(ok ? (sign | ((unsigned int)(E - 896) << 23) | m23) : out_of_range);
  const unsigned int r29 = (unsigned int)b & 0x1FFFFFFFu;
  // scale 2^(E-1075) as a float: exponent field E - 948 (0 below 2^-74)
  const float scale = __int_as_float(E >= 949 ? ((unsigned int)(E - 948) << 23) : 0u);
  const float l = __uint2float_rn(r29) * scale;
  lo = ok ? (sign ? -l : l) : 0.f;
}
// Debug-bounds build (-DFK_DEBUG_BOUNDS): the step kernel checks the index
// of each shared- and global-memory access and of each bulk copy against its
// buffer first; a failed check sets kFlagBounds in the grid's state and the
// access is skipped (a skipped copy still completes its stage's phase).  In
// the release build every check is the constant true.
#ifdef FK_DEBUG_BOUNDS
__device__ __forceinline__ bool in_bounds(bool ok, DevState* st) {
  if (!ok) atomicOr(&st->flags, kFlagBounds);
  return ok;
}
#else
__device__ __forceinline__ constexpr bool in_bounds(bool, DevState*) { return true; }
#endif

// s + c += x, exactly in s (TwoSum), the rounding error collected in c
__device__ __forceinline__ void two_sum_acc(float& s, float& c, float x) {
  const float t = s + x;
  const float bp = t - s;
  c += (s - (t - bp)) + (x - bp);
  s = t;
}

// FP32 pairs x.x + x.y, for the wall sums of FP32 grids' half units:
// the leading product of a pair by a float or a pair is exact (TwoProd
// with a fused multiply-add), sums take TwoSum of the leading parts and add
// the trailing parts (Dekker 1971; Knuth, TAOCP Vol. 2, 4.2.2), about 44
// bits in all, on the FP32 pipe instead of GB300's narrow FP64 one.
__device__ __forceinline__ float2 pair_mul(float2 a, float b) {
  const float p = a.x * b;
  float e = fmaf(a.x, b, -p);
  e = fmaf(a.y, b, e);
  return make_float2(p, e);
}
__device__ __forceinline__ float2 pair_mul(float2 a, float2 b) {
  const float p = a.x * b.x;
  float e = fmaf(a.x, b.x, -p);
  e = fmaf(a.x, b.y, e);
  e = fmaf(a.y, b.x, e);
  return make_float2(p, e);
}
__device__ __forceinline__ void pair_acc(float2& s, float2 x) {
  two_sum_acc(s.x, s.y, x.x);
  s.y += x.y;
}
// sum over the warp, valid in lane 0
__device__ __forceinline__ float2 pair_warp_sum(float2 v) {
  for (int o = 16; o > 0; o >>= 1) {
    const float oh = __shfl_down_sync(0xffffffffu, v.x, o);
    const float ol = __shfl_down_sync(0xffffffffu, v.y, o);
    two_sum_acc(v.x, v.y, oh);
    v.y += ol;
  }
  return v;
}

// Coefficients of one pipeline item (resident kernel).
struct ItemVals {
  double a1;             // |c_1| (FP64 grids)
  float c1, bgk_a, bgk_s;  // c_1; dt nu and dt nu n (FP32 grids)
  float pad;
};

// Wall (x = 0, v1 < 0: Eqs. 12-14) or vacuum (x = h_max, v1 > 0) sums of
// f^{n+1} over this consumer thread's cells of one plane, read back from
// its own stores; returns whether one of those cells is negative.  Called
// only on those two planes of a march, so the main loop carries no FP64
// instruction for them.  Two FP64 operations a cell on the wall (the yield
// comes multiplied by -v1), one on the vacuum side.
template <typename T>
__device__ __noinline__ bool wall_terms(const T* oplane, const double* v1tab,
                                        const double* vdelta, int tid, int nthreads, int i0,
                                        int rows, int nv2, int pitch, bool wall, double* out3) {
  constexpr int VEC = 16 / sizeof(T);
  const int QV = pitch / VEC;
  double pe = 0.0, see = 0.0, vac = 0.0;
  bool neg = false;
  for (int m = 0; m < kVecPerThread; m++) {
    const int v = tid + nthreads * m;
    if (v >= rows * QV) break;
    const int r = v / QV, q = v - (v / QV) * QV;
    const int i = i0 + r;
    const double v1 = v1tab[i];
    for (int e = 0; e < VEC && q * VEC + e < nv2; e++) {
      const size_t c = (size_t)i * pitch + q * VEC + e;
      const T f = oplane[c];
      neg = neg || is_negative(f);
      const double fn = (double)f;
      if (wall) {
        pe = fma(-v1, fn, pe);         // Eq. 13 without dv1 dv2
        see = fma(vdelta[c], fn, see);  // Eq. 12
      } else {
        vac = fma(v1, fn, vac);
      }
    }
  }
  out3[0] = pe;
  out3[1] = see;
  out3[2] = vac;
  return neg;  // a value of the plane is negative
}

// The same sums for the half-CTA units of FP32 grids, in FP32 pairs (v1
// and delta as pairs, exact leading products) and folded over the warp
// (out3 valid in lane 0): thin tiles run three CTAs to an SM, and there the
// FP64 instructions of the two boundary planes held up whole units.
__device__ __noinline__ bool wall_terms_pairs(const float* oplane, const float2* v1p,
                                              const float2* deltap, int tid, int nthreads,
                                              int i0, int rows, int nv2, int pitch, bool wall,
                                              double* out3) {
  const int QV = pitch / 4;
  float2 pe = make_float2(0.f, 0.f), see = pe, vac = pe;
  bool neg = false;
  for (int m = 0; m < kVecPerThread; m++) {
    const int v = tid + nthreads * m;
    if (v >= rows * QV) break;
    const int r = v / QV, q = v - (v / QV) * QV;
    const int i = i0 + r;
    const float2 v1 = v1p[i];
    for (int e = 0; e < 4 && q * 4 + e < nv2; e++) {
      const size_t c = (size_t)i * pitch + q * 4 + e;
      const float fn = oplane[c];
      neg = neg || fn < 0.f;
      const float2 g = pair_mul(v1, fn);
      if (wall) {
        const float2 mg = make_float2(-g.x, -g.y);  // Eq. 13 without dv1 dv2
        pair_acc(pe, mg);
        pair_acc(see, pair_mul(deltap[c], mg));  // Eq. 12
      } else {
        pair_acc(vac, g);
      }
    }
  }
  pe = pair_warp_sum(pe);
  see = pair_warp_sum(see);
  vac = pair_warp_sum(vac);
  out3[0] = (double)pe.x + (double)pe.y;
  out3[1] = (double)see.x + (double)see.y;
  out3[2] = (double)vac.x + (double)vac.y;
  return neg;  // a value of the thread's cells is negative
}

// wall_terms and wall_terms_pairs (PAIRS) for the resident kernel, where the
// boundary plane is the last one of a march and its sums are on the way of
// the next step: the same sums in the same order, inline after the march
// (whose registers are free by then), with the loads of B vectors at a time
// ahead of the arithmetic.  One load after another, as in the helpers above,
// took as long as four planes.  Row padding holds zeros of f and delta.
template <typename T, bool PAIRS>
__device__ __forceinline__ bool wall_terms_ahead(const T* oplane, const Tables& tab, int tid,
                                                 int nthreads, int i0, int rows, int pitch,
                                                 bool wall, double* out3) {
  constexpr int VEC = 16 / sizeof(T);
  constexpr int B = 2;
  // v1 and delta as pairs, or v1 and -v1 delta in FP64
  using W = std::conditional_t<PAIRS, float2, double>;
  const W* v1tab;
  const W* deltab;
  if constexpr (PAIRS) {
    v1tab = tab.v1p;
    deltab = tab.deltap;
  } else {
    v1tab = tab.v1;
    deltab = tab.vdelta;
  }
  const int QV = pitch / VEC, nv = rows * QV;
  float2 pe2 = make_float2(0.f, 0.f), see2 = pe2, vac2 = pe2;
  double pe = 0.0, see = 0.0, vac = 0.0;
  bool neg = false;
  for (int m0 = 0; m0 < kVecPerThread && nthreads * m0 < nv; m0 += B) {
    float4 f[B];
    W v1[B];
    float4 d[B][VEC / 2];  // 2 of W in each
#pragma unroll
    for (int b = 0; b < B; b++) {
      const int v = tid + nthreads * (m0 + b);
      const int r = v < nv ? v / QV : 0;
      const size_t c = (size_t)(i0 + r) * pitch + (v < nv ? (v - r * QV) * VEC : 0);
      f[b] = __ldcg(reinterpret_cast<const float4*>(oplane + c));
      v1[b] = v1tab[i0 + r];
#pragma unroll
      for (int e = 0; e < VEC / 2; e++)
        d[b][e] = wall ? reinterpret_cast<const float4*>(deltab + c)[e] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int b = 0; b < B; b++) {
      if (tid + nthreads * (m0 + b) >= nv) break;
      const Vec<T> fv = *reinterpret_cast<const Vec<T>*>(&f[b]);
      const W* dv = reinterpret_cast<const W*>(&d[b][0]);
#pragma unroll
      for (int e = 0; e < VEC; e++) {
        neg = neg || is_negative(fv.e[e]);
        if constexpr (PAIRS) {
          const float2 g = pair_mul(v1[b], (float)fv.e[e]);
          if (wall) {
            const float2 mg = make_float2(-g.x, -g.y);  // Eq. 13 without dv1 dv2
            pair_acc(pe2, mg);
            pair_acc(see2, pair_mul(dv[e], mg));  // Eq. 12
          } else {
            pair_acc(vac2, g);
          }
        } else {
          const double fn = (double)fv.e[e];
          if (wall) {
            pe = fma(-v1[b], fn, pe);
            see = fma(dv[e], fn, see);
          } else {
            vac = fma(v1[b], fn, vac);
          }
        }
      }
    }
  }
  if constexpr (PAIRS) {  // folded over the warp, valid in lane 0
    pe2 = pair_warp_sum(pe2);
    see2 = pair_warp_sum(see2);
    vac2 = pair_warp_sum(vac2);
    pe = (double)pe2.x + (double)pe2.y;
    see = (double)see2.x + (double)see2.y;
    vac = (double)vac2.x + (double)vac2.y;
  } else {
    pe = warp_sum(pe);
    see = warp_sum(see);
    vac = warp_sum(vac);
  }
  out3[0] = pe;
  out3[1] = see;
  out3[2] = vac;
  return neg;
}

// Barrier over the threads of one unit: the whole CTA (barrier 0), or one
// half of it (named barrier 1 or 2, kHalfBlock threads).
template <int NT>
__device__ __forceinline__ void unit_sync(int bar) {
  if constexpr (NT == kThreads) {
    __syncthreads();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NT + 32) : "memory");
  }
}

// A pointer field of the step arguments read where it is used.  SA: the
// arguments sit in the CTA's shared memory (batched kernels), and a read
// there at each use (an LDS) keeps the pointer out of the registers of the
// march; otherwise they are kernel parameters, which instructions take
// directly.
template <bool SA, typename X>
__device__ __forceinline__ X arg_at_use(const X& field) {
  static_assert(sizeof(X) == 8, "pointer fields");
  if constexpr (SA) {
    unsigned long long v;
    asm volatile("ld.shared.b64 %0, [%1];"
                 : "=l"(v)
                 : "r"((unsigned)__cvta_generic_to_shared(&field)));
    return reinterpret_cast<X>(v);
  } else {
    return field;
  }
}

// One unit (tile t, chunk) of a grid on NT consumer threads (kThreads, or
// kHalfThreads for a half-CTA unit) plus a producer warp; tid: the thread's
// index within the unit, bar: the unit's barrier; smem is the unit's shared
// memory past its argument slot.  BGK: the grid has the electron-electron
// collision term of Eq. 3 switched on.  SA: a is in shared memory.
// RES: the unit's part of rs.n_steps steps (resident step kernel), else of one.
template <typename T, bool PADDED, bool BGK, int NT, bool SA, bool RES = false>
__device__ __forceinline__ void stream_unit(const StepArgs& a, const int t, const int chunk,
                                            unsigned char* smem, const int tid, const int bar,
                                            const Resident& rs = Resident()) {
  constexpr int NW = NT / 32;  // consumer warps
  constexpr int NS = unit_stages<NT>();  // stages of the ring
  constexpr int VEC = Vec<T>::N;
  constexpr int M = unit_vectors<NT, (int)sizeof(T)>();
  // per-plane pointer reads from the shared-memory arguments at their use
  // where the march runs out of registers (half units, FP64 grids with
  // collisions); elsewhere the pointers stay in registers (measured faster;
  // FP32 batches with collisions spilled 20 bytes with them read at use and
  // none without: four grids of 1024 x 128 x 128 139 -> 132 us a step)
  constexpr bool SAU = SA && (NT == kHalfThreads || (BGK && sizeof(T) == 8));
  // compact index arithmetic (an item's plane in one multiply-add, 32-bit
  // stage and plane sizes), where it keeps the march's registers within the
  // launch bounds: without it the plain whole-CTA FP32 batch kernel spills 40
  // bytes in the march, and three grids of 1024 x 256 x 256 take 318 us a
  // launch instead of 263 (0.745 and 0.90 of copy bandwidth).  The other plain
  // whole-CTA kernels do without: a grid alone has no spill either way (with it
  // 104 us instead of 99.7 at 1024 x 256 x 256, 49 instead of 52 at 600 x 200 x
  // 200), the FP64 and the resident ones spill less.
  constexpr bool COMPACT = NT == kHalfThreads || PADDED || BGK || (SA && sizeof(T) == 4);
  using StageSz = std::conditional_t<COMPACT, unsigned, size_t>;  // < 227 KB
  using PlaneSz = std::conditional_t<COMPACT, int, size_t>;
  const Geom& gm = a.geom;
  const StageSz sbytes = (StageSz)stage_bytes<T>(gm.stage_elems);
  unsigned char* stage_base = smem;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NS * sbytes);
  uint64_t* empty = full + NS;
  double* wsum = reinterpret_cast<double*>(empty + NS);  // [NS][kWarps][kWs]
  double* dgl = wsum + NS * kWarps * kWs;  // [NS][kMaxTileRows], FP64
  float* srow_s = reinterpret_cast<float*>(dgl);  // [kMaxTileRows], FP32
  float* scol_s = srow_s + kMaxTileRows;          // [pitch], FP32
  unsigned char* bgk_base = reinterpret_cast<unsigned char*>(dgl) + tail_main_bytes<T, NS>(a.pitch);
  double* dgs = reinterpret_cast<double*>(bgk_base);  // [NS][kMaxTileRows], FP64
  double* m2d = dgs + NS * kMaxTileRows;         // [pitch], FP64
  float* m1_s = reinterpret_cast<float*>(bgk_base);   // [kMaxTileRows], FP32
  float* m2_s = m1_s + kMaxTileRows;                  // [pitch], FP32
  // control words (RES: ctl[4] is set when a wait of the unit runs out, ctl[5]
  // when no further step follows; then what the consumers need of the item in
  // each stage, read from L2 once, by the producer)
  int* ctl = reinterpret_cast<int*>(bgk_base + tail_bgk_bytes<T, NS>(a.pitch));
  ItemVals* iv = reinterpret_cast<ItemVals*>(ctl + 8);

  const int lane = tid & 31, warp = tid >> 5;
  const int nt = gm.n_tiles;
  const int nx = a.nx, nv1 = a.nv1, nv2 = a.nv2, pitch = a.pitch;
  int i0, i1, dir;
  tile_rows(gm, nv1, t, &i0, &i1, &dir);
  // (a launch of many steps starts with a shorter chunk)
  const int s0 = RES ? max(0, chunk * gm.chunk_len - gm.chunk_off) : chunk * gm.chunk_len;
  const int s1 = RES ? min(nx, (chunk + 1) * gm.chunk_len - gm.chunk_off)
                     : min(nx, s0 + gm.chunk_len);
  if (s0 >= s1 || i0 >= i1) return;  // uniform over the block
  // the tile fits its row tables and a stage holds it with its halo row
  if (!in_bounds(i0 >= 0 && i1 <= nv1 && i1 - i0 <= kMaxTileRows &&
                     (i1 - i0 + 1) * pitch <= gm.stage_elems,
                 a.st))
    return;  // uniform over the block

  // march: step s visits plane k(s); the upwind plane of the first one is
  // loaded first ("prime" item) unless it lies outside the domain
  const int k_first = dir > 0 ? s0 : nx - 1 - s0;
  const int k_up = k_first - dir;
  const bool prime = k_up >= 0 && k_up < nx;
  const int n_items = (s1 - s0) + (prime ? 1 : 0);
  // item q visits plane k_first + dir (q - 1) after a prime item (q = 0:
  // k_up), plane k_first + dir q without one
  const int k_item0 = prime ? k_up : k_first;
  auto item_plane = [&](int q) -> int {
    if constexpr (COMPACT) {
      return k_item0 + dir * q;
    } else {
      const int s = s0 + q - (prime ? 1 : 0);
      if (s < s0) return k_up;
      return dir > 0 ? s : nx - 1 - s;
    }
  };

  if (sizeof(T) == 4) {  // source factors of this tile (FP32 grids)
    for (int r = tid; r < i1 - i0; r += NT + 32) srow_s[r] = a.tab.srow32[i0 + r];
    for (int j = tid; j < pitch; j += NT + 32) scol_s[j] = a.tab.scol32[j];
  }
  if (BGK) {  // factors of the collision equilibrium (Eq. 5)
    if (sizeof(T) == 4) {
      for (int r = tid; r < i1 - i0; r += NT + 32) m1_s[r] = a.tab.m1_32[i0 + r];
      for (int j = tid; j < pitch; j += NT + 32) m2_s[j] = a.tab.m2_32[j];
    } else {
      for (int j = tid; j < pitch; j += NT + 32) m2d[j] = a.tab.m2[j];
    }
  }
  long long* wlim = reinterpret_cast<long long*>(ctl + 2);  // bounded waits' limit (cycles)
  if (tid == 0) {
    ctl[0] = (int)ld_shared_value<RES>(&a.st->flags);
    if constexpr (RES) ctl[4] = ctl[5] = 0;
    // test knob: the pipeline item whose copy this unit does not issue
    ctl[1] = (t == 0 && chunk == 0) ? a.prm->withhold_item : -1;
    *wlim = a.prm->wait_limit;
    for (int s = 0; s < NS; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], NT);
    }
    fence_mbar_init();
  }
  unit_sync<NT>(bar);
  if (ctl[0]) {  // sticky error: freeze the state (uniform)
    if constexpr (RES)
      if (tid == 0) count_arrival(rs.arrive, 1);
    return;
  }

  const Params& p = *a.prm;
  using InPtr = std::conditional_t<RES, const T*, const T* __restrict__>;
  using OutPtr = std::conditional_t<RES, T*, T* __restrict__>;
  InPtr fin = static_cast<const T*>(a.f_in);
  OutPtr fout = static_cast<T*>(a.f_out);
  // RES: the unit's end of step s -- its threads' stores, then one arrival
  auto end_step = [&]() {
    fence_proxy_async_global();
    unit_sync<NT>(bar);
    if (tid == 0) count_arrival(rs.arrive, 1);
  };
  // RES: wait until the launch's counter reaches `want`; false if it says stop
  // (or the wait runs out: the step is lost)
  auto wait_count = [&](const unsigned* counter, unsigned want) -> bool {
    const long long lim = *wlim, t0 = clock64();
    unsigned v = read_count(counter);
    while (v < want) {
      if (clock64() - t0 > lim) {
        atomicOr(&a.st->flags, kFlagTimeout);
        return false;
      }
      v = read_count(counter);
    }
    return v < kGoStop;
  };
  // cells of a plane (below 2^31, as a streamed row holds at most one
  // unit's cells, 7168, and nv1 <= 65536)
  const PlaneSz plane = (PlaneSz)nv1 * pitch;
  const int QV = pitch / VEC;  // vectors per row
  const int stage_n = gm.stage_elems;     // elements of a stage
  const size_t f_n = (size_t)nx * plane;  // elements of f
  const int rows = i1 - i0;

  if (warp == NW) {
    // ============================ producer warp ============================
    // Per item q: wait until every consumer released the stage of item
    // q - NS, read what its partial sums need from that stage and from
    // the warp sums (gather), refill the stage with item q (issue), then
    // reduce and store the partial sums of item q - NS (finish): the
    // reductions run while the copy is in flight.
    //
    // c_1 (FP32 copy) of item q sits in lane q % 32 of c1w (items wbase ..
    // wbase + 31) or of c1n (the next 32 items, loaded a window ahead);
    // lane st of c1slot / a1slot holds c_1 and |c_1| (FP64 grids) of the
    // item in stage st.
    const T a2t = (T)fabs(p.c2);
    const bool has_a2 = p.c2 != 0.0;
    int it0 = 0;  // RES: items of the steps before (the ring runs on through them)
    // RES: with the collision coefficients and FP64 |c_1| beside it
    struct Window {
      float c1;
      T a1, ba, bs;
    };
    auto load_window = [&](int base) -> Window {
      Window w{0.f, (T)0, (T)0, (T)0};
      if (base + lane < n_items) {
        const int k = item_plane(base + lane);
        w.c1 = ld_shared_value<RES>(a.c1_32 + k);
        if constexpr (RES && sizeof(T) == 8) {
          w.a1 = fabs(__ldcg(a.c1 + k));
          if (BGK) {
            w.ba = __ldcg(a.bgk + k);
            w.bs = __ldcg(a.bgk + nx + k);
          }
        } else if constexpr (RES && BGK) {
          w.ba = __ldcg(a.bgk32 + k);
          w.bs = __ldcg(a.bgk32 + nx + k);
        }
      }
      return w;
    };
    Window ww, wn;  // this window of 32 items and the next
    float c1first;  // c_1 of items 0 .. 31 of the step
    int wbase;
    auto first_window = [&]() {
      ww = load_window(0);
      wn = load_window(32);
      wbase = 0;
      c1first = ww.c1;
    };
    first_window();
    const int n_pre = min(NS, n_items);  // RES: items fetched ahead of a step
    // RES, FP64 grids: the diagonal's part that no plane changes
    double d0[2] = {0.0, 0.0};
    if constexpr (RES && sizeof(T) == 8)
      for (int h = 0; h < 2; h++)
        if (lane + 32 * h < rows) d0[h] = (1.0 - fabs(p.c2)) - fabs(a.tab.cx[i0 + lane + 32 * h]);
    float c1slot = 0.f;
    double a1slot = 0.0;
    // What the sums and (FP64 grids) the consumers need to know of item q,
    // whose plane has the v1-Courant number c1
    auto set_item = [&](int q, float c1) {
      const int k = item_plane(q);
      const int st = (it0 + q) % NS;
      if (lane == st) c1slot = c1;
      if (sizeof(T) == 8) {
        // FP64 diagonal of the convex update per tile row, once per plane
        // here rather than per vector in the consumers: (1 - |c_2| - |c_x|)
        // less |c_1| and the loss part of the collision term, dt nu_k f
        double a1, ba = 0.0, bs = 0.0;
        if constexpr (RES) {
          a1 = __shfl_sync(0xffffffffu, ww.a1, q & 31);
          if (c1 == 0.f) a1 = 0.0;
          if (BGK) {
            ba = __shfl_sync(0xffffffffu, ww.ba, q & 31);
            bs = __shfl_sync(0xffffffffu, ww.bs, q & 31);
          }
          if (lane == 0) iv[st].a1 = a1;
        } else {
          a1 = c1 == 0.f ? 0.0 : fabs(a.c1[k]);
          if (BGK) {
            ba = a.bgk[k];
            bs = a.bgk[nx + k];
          }
        }
        if (lane == st) a1slot = a1;
        const double loss = BGK ? a1 + ba : a1;
        for (int h = 0; h < 2; h++) {
          const int r = lane + 32 * h;
          if (r >= rows) break;
          const double d = RES ? d0[h] : (1.0 - fabs(p.c2)) - fabs(a.tab.cx[i0 + r]);
          dgl[st * kMaxTileRows + r] = d - loss;
          // the gain part of the collision term per tile row: dt nu_k n_k m1[i]
          if (BGK) dgs[st * kMaxTileRows + r] = bs * a.tab.m1[i0 + r];
        }
      }
      if constexpr (RES) {
        const float ba = BGK ? (float)__shfl_sync(0xffffffffu, ww.ba, q & 31) : 0.f;
        const float bs = BGK ? (float)__shfl_sync(0xffffffffu, ww.bs, q & 31) : 0.f;
        if (lane == 0) {
          iv[st].c1 = c1;
          if (sizeof(T) == 4) {
            iv[st].bgk_a = ba;
            iv[st].bgk_s = bs;
          }
        }
      }
    };
    // all 32 lanes: where the upwind v1 halo row lies outside the velocity
    // grid, fill its slot with zeros (zero inflow through the v1 edge) so
    // the consumers read a neighbour row without a bounds test.
    // stage layout: the tile's rows start at row 1 when the halo lies
    // above (c_1 > 0), at row 0 otherwise (halo, if any, at row `rows`)
    auto zero_halo = [&](T* stage, float c1) {
      int zrow = -1;
      if (c1 > 0.f && i0 == 0) zrow = 0;
      if (c1 < 0.f && i1 == nv1) zrow = rows;
      if (zrow >= 0 && in_bounds((zrow + 1) * pitch <= stage_n, a.st)) {
        float4* z = reinterpret_cast<float4*>(stage + (size_t)zrow * pitch);
        const int n16 = pitch * (int)sizeof(T) / 16;
        for (int c = lane; c < n16; c += 32) z[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        // a later bulk copy (async proxy) may land on these bytes when c_1
        // changes sign: order the zero stores (generic proxy) before it
        fence_proxy_async_smem();
      }
    };
    // The span of f that plane k's stage takes: the tile's rows plus the halo
    // row inside the grid; its elements, where it starts in the stage and in f
    auto item_span = [&](int k, float c1, int* dofs, size_t* sofs) -> int {
      int lo = i0, hi = i1;
      if (c1 > 0.f && i0 > 0) lo = i0 - 1;  // v1 halo row on the upwind side
      if (c1 < 0.f && i1 < nv1) hi = i1 + 1;
      *dofs = (lo - i0 + (c1 > 0.f ? 1 : 0)) * pitch;
      *sofs = (size_t)k * plane + (size_t)lo * pitch;
      const int n = (hi - lo) * pitch;
      return in_bounds(k >= 0 && k < nx && lo >= 0 && hi <= nv1 && *dofs >= 0 &&
                           *dofs + n <= stage_n && *sofs + (size_t)n <= f_n,
                       a.st)
                 ? n
                 : 0;
    };
    // the zero row, then lane 0 copies plane k's span
    auto issue_copy = [&](int q, float c1) {
      const int k = item_plane(q);
      const int st = (it0 + q) % NS;
      T* stage = reinterpret_cast<T*>(stage_base + st * sbytes);
      zero_halo(stage, c1);
      __syncwarp();
      if (lane == 0 && it0 + q != ctl[1]) {  // ctl[1]: a withheld item (test knob), else -1
        int dofs;
        size_t sofs;
        const uint32_t bytes = (uint32_t)(item_span(k, c1, &dofs, &sofs) * (int)sizeof(T));
        if (bytes) {
          mbar_expect_tx(&full[st], bytes);  // release: the zero row is visible too
          bulk_g2s(stage + dofs, fin + sofs, bytes, &full[st]);
        } else {
          mbar_expect_tx(&full[st], 0);  // no data: the stage's phase completes
        }
      }
    };
    auto issue = [&](int q) {
      if (q == wbase + 32) {  // next window; prefetch the one after
        ww = wn;
        wbase += 32;
        wn = load_window(wbase + 32);
      }
      const float c1 = __shfl_sync(0xffffffffu, ww.c1, q & 31);
      set_item(q, c1);
      issue_copy(q, c1);
    };
    // RES: item q's plane was copied for a c_1 of another sign than its own:
    // lay the stage out anew, with plain loads (rare: E_x of the plane changed
    // its sign in this step)
    auto lay_out_again = [&](int q, float c1) {
      const int st = (it0 + q) % NS;
      T* stage = reinterpret_cast<T*>(stage_base + st * sbytes);
      if (!__all_sync(0xffffffffu,
                      mbar_wait(&full[st], (uint32_t)(((it0 + q) / NS) & 1), wlim))) {
        if (lane == 0) {
          atomicOr(&a.st->flags, kFlagTimeout);
          ctl[5] = 1;
        }
        return;
      }
      int dofs;
      size_t sofs;
      const int n16 = item_span(item_plane(q), c1, &dofs, &sofs) / VEC;
      const float4* src = reinterpret_cast<const float4*>(fin + sofs);
      float4* dst = reinterpret_cast<float4*>(stage + dofs);
      for (int c = lane; c < n16; c += 32) dst[c] = __ldcg(src + c);
      zero_halo(stage, c1);
      fence_proxy_async_smem();
    };
    // What the partial sums of a consumed compute item need from its stage
    // and from the warp sums, read before the stage is refilled.
    struct Gathered {
      int k;       // plane (-1: the prime item, no sums)
      T lvt;       // this lane's share of the velocity-edge outflow
      float2 wsf;  // lane w < NW: warp w's density sum (FP64 grids: hi, lo)
      double ws[kWs];  // lane w < NW: warp w's other sums, on a wall plane
    };
    auto gather = [&](int q) -> Gathered {
      Gathered g;
      g.k = -1;
      g.lvt = (T)0;
      g.wsf = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < kWs; i++) g.ws[i] = 0.0;
      if (prime && q == 0) return g;
      const int k = item_plane(q);
      const int st = (it0 + q) % NS;
      g.k = k;
      const T* sb = reinterpret_cast<const T*>(stage_base + st * sbytes);
      const float c1f = __shfl_sync(0xffffffffu, c1slot, st);
      const double a1d = sizeof(T) == 8 ? __shfl_sync(0xffffffffu, a1slot, st) : 0.0;
      // ledger: outflow of f^n through the downwind velocity edges, summed
      // in the grid's precision (a ledger diagnostic: FP32 grids keep FP64
      // instructions off this per-plane path)
      const T a1t = sizeof(T) == 4 ? (T)fabsf(c1f) : (T)a1d;
      const int erow = (c1f > 0.f && i1 == nv1) ? nv1 - 1 : ((c1f < 0.f && i0 == 0) ? 0 : -1);
      const int rb = c1f > 0.f ? 1 : 0;  // stage row of the tile's first row
      if (erow >= 0 && in_bounds(erow - i0 + rb >= 0 && (erow - i0 + rb + 1) * pitch <= stage_n,
                                 a.st)) {
        const T* r = sb + (size_t)(erow - i0 + rb) * pitch;
        for (int j = lane; j < nv2; j += 32) g.lvt += a1t * r[j];
      }
      if (has_a2 && in_bounds((rows - 1 + rb) * pitch + nv2 <= stage_n, a.st))
        for (int r = lane; r < rows; r += 32) g.lvt += a2t * sb[(size_t)(r + rb) * pitch + nv2 - 1];
      if (lane < NW) {
        const double* ws = wsum + (st * kWarps + lane) * kWs;
        if constexpr (sizeof(T) == 4)
          g.wsf.x = *reinterpret_cast<const float*>(ws);
        else
          g.wsf = *reinterpret_cast<const float2*>(ws);
        if (k == 0 || k == nx - 1) {
#pragma unroll
          for (int i = 1; i < kWs; i++) g.ws[i] = ws[i];
        }
      }
      return g;
    };
    double* lvp = a.part.lv;
    // fold the gathered sums (the warps' in a fixed order) and store them
    auto finish = [&](const Gathered& g) {
      if (g.k < 0) return;
      const int k = g.k;
      const double lv = (double)warp_sum(g.lvt);
      double sum[kWs] = {0.0, 0.0, 0.0, 0.0};
      const bool wall = k == 0 || k == nx - 1;
      if constexpr (sizeof(T) == 4) {  // added in FP32, one conversion per plane
        float sumf = 0.f;
#pragma unroll
        for (int w = 0; w < NW; w++) sumf += __shfl_sync(0xffffffffu, g.wsf.x, w);
        sum[0] = (double)sumf;
      } else {
        // An FP64 instruction takes the SM's FP64 pipe 16 cycles, for one lane
        // as for 32, and that pipe bounds FP64 grids: the warps' pairs become
        // FP64 here, all at once, and are folded in a tree.  With the
        // conversions in each consumer warp and a serial fold a plane of 13 rows
        // of 256 took 40 FP64 instructions beside its 416 for the update: 603 us
        // a step at 1024 x 256 x 256, now 574; 512 x 128 x 128 92 -> 88 us.
        sum[0] = (double)g.wsf.x + (double)g.wsf.y;
#pragma unroll
        for (int o = NW > 4 ? 4 : 2; o > 0; o >>= 1)
          sum[0] += __shfl_down_sync(0xffffffffu, sum[0], o);
      }
      if (wall) {
#pragma unroll
        for (int w = 0; w < NW; w++)
#pragma unroll
          for (int i = 1; i < kWs; i++) sum[i] += __shfl_sync(0xffffffffu, g.ws[i], w);
      }
      if (lane == 0 && in_bounds(k >= 0 && k < nx && t >= 0 && t < nt, a.st)) {
        a.part.n[(size_t)k * nt + t] = sum[0];
        lvp[(size_t)k * nt + t] = lv;
        if (k == 0) {
          a.part.pe[t] = sum[1];
          a.part.see[t] = sum[2];
        }
        if (k == nx - 1) a.part.vac[t] = sum[3];
      }
    };
    const int n_steps = RES ? rs.n_steps : 1;
    for (int step = 0; step < n_steps; step++) {
      if constexpr (RES) {
        if (step > 0) {
          // the new state is whole: fetch the first planes, laid out for the
          // last step's c_1, while the finalize runs
          if (lane == 0 && !wait_count(rs.arrive, rs.n_units * (unsigned)step)) ctl[5] = 1;
          __syncwarp();
          InPtr x = fout;
          fout = const_cast<T*>(fin);
          fin = x;
          it0 += n_items;
          lvp = step & 1 ? rs.lv_odd : a.part.lv;
          const float guess = c1first;
          const bool fetch = ctl[5] == 0;
          if (fetch) {
            fence_proxy_async_global();
            for (int q = 0; q < n_pre; q++) issue_copy(q, __shfl_sync(0xffffffffu, guess, q));
            if (lane == 0 && !wait_count(rs.go, rs.n_fin * (unsigned)step)) ctl[5] = 1;
            __syncwarp();
            if (ctl[5] == 0) {
              first_window();
              for (int q = 0; q < n_pre; q++) {
                const float c1 = __shfl_sync(0xffffffffu, c1first, q);
                const float was = __shfl_sync(0xffffffffu, guess, q);
                if ((c1 > 0.f) != (was > 0.f) || (c1 < 0.f) != (was < 0.f)) lay_out_again(q, c1);
                set_item(q, c1);
              }
            }
            __syncwarp();
            if (ctl[5])  // the copies in flight land before the CTA leaves
              for (int q = 0; q < n_pre; q++)
                mbar_wait(&full[(it0 + q) % NS], (uint32_t)(((it0 + q) / NS) & 1), wlim);
          }
          unit_sync<NT>(bar);
          if (ctl[5]) return;
        }
      }
      int issued = 0;
      bool ok = true;
      for (int q = 0; q < n_items; q++) {
        Gathered g{};
        g.k = -1;
        if (q >= NS) {
          // stage reuse: wait until every consumer thread released item q - NS
          ok = __all_sync(0xffffffffu, mbar_wait(&empty[(it0 + q) % NS],
                                                 (uint32_t)((((it0 + q) / NS) - 1) & 1), wlim));
          if (!ok) break;
          g = gather(q - NS);
          __syncwarp();  // the stage is read by every lane before it is refilled
        }
        if (!RES || step == 0 || q >= n_pre) issue(q);
        issued = q + 1;
        finish(g);
      }
      for (int q = max(0, issued - NS); q < issued && ok; q++) {
        ok = __all_sync(0xffffffffu, mbar_wait(&empty[(it0 + q) % NS],
                                               (uint32_t)(((it0 + q) / NS) & 1), wlim));
        if (ok) finish(gather(q));
      }
      if (!ok && lane == 0) {
        atomicOr(&a.st->flags, kFlagTimeout);
        if constexpr (RES) ctl[4] = 1;
        // copies still in flight land before the CTA leaves (a withheld
        // item's copy was never issued: nothing to wait for)
        for (int q = max(0, issued - NS); q < issued; q++)
          if (it0 + q != ctl[1])
            mbar_wait(&full[(it0 + q) % NS], (uint32_t)(((it0 + q) / NS) & 1), wlim);
      }
      if constexpr (RES) {
        end_step();
        if (ctl[4]) return;
      }
    }
    return;
  }

  // ============================ consumer warps =============================
  // this thread's cells: vectors v = tid + NT*m of the tile, fixed for
  // the whole march; per vector its offset in a stage and in a plane
  int soff[M];  // offset from the tile's first cell (low 24 bits) and row (top byte)
  const int gbase = i0 * pitch;  // the tile's first cell in a plane
  // bit m: vector m exists / starts a row; zleft bit 16 + m: vector m is
  // the last of a padded row (pitch > nv2: only a row's last vector holds
  // padding, its elements from nv2 - (pitch - VEC) on)
  unsigned valid = 0, zleft = 0;
  T ax[M];
  T xr[M][VEC];
#pragma unroll
  for (int m = 0; m < M; m++) {
    const int v = tid + NT * m;
    // a vector past the tile reads its first cells instead and writes nothing
    soff[m] = 0;
    ax[m] = (T)0;
    if (v >= rows * QV) {
      zleft |= 1u << m;
    } else {
      const int r = v / QV, qv = v - r * QV;
      valid |= 1u << m;
      if (qv == 0) zleft |= 1u << m;
      if (PADDED && qv == QV - 1 && pitch != nv2) zleft |= 1u << (16 + m);
      soff[m] = (r * pitch + qv * VEC) | (r << 24);
      const T cx = sizeof(T) == 8 ? (T)a.tab.cx[i0 + r] : (T)a.tab.cx32[i0 + r];
      ax[m] = cx < (T)0 ? -cx : cx;
    }
#pragma unroll
    for (int e = 0; e < VEC; e++) xr[m][e] = (T)0;
  }
  // the x-upwind values of a march's first plane
  auto first_upwind = [&]() {
    if (!prime && dir > 0) {
      // first plane is x = 0 with v1 > 0: the upwind value is the re-emitted
      // distribution Gamma_see g_se of Eq. 15 (zero for the vacuum side)
      // (plus, with reflection, refl times the incident f^n of the mirror
      // cell at -v1 on the same plane)
      const double gsee = ld_shared_value<RES>(&a.st->g_see);
      const double refl = p.refl;
#pragma unroll
      for (int m = 0; m < M; m++) {
        if (!(valid >> m & 1)) continue;
        const int r = soff[m] >> 24;
        const int c0 = (soff[m] & 0xFFFFFF) - r * pitch;
        if constexpr (!RES) {
#pragma unroll
          for (int e = 0; e < VEC; e++) {
            double g = gsee * a.tab.gse[(soff[m] & 0xFFFFFF) + gbase + e];
            if (refl > 0.0)
              g = fma(refl, (double)fin[(size_t)(nv1 - 1 - (i0 + r)) * pitch + c0 + e], g);
            xr[m][e] = (T)g;
          }
        } else {  // the same with vector loads
          const double2* g2 =
              reinterpret_cast<const double2*>(a.tab.gse + (soff[m] & 0xFFFFFF) + gbase);
          double g[VEC];
#pragma unroll
          for (int e = 0; e < VEC; e += 2) {
            const double2 x = __ldg(g2 + e / 2);
            g[e] = gsee * x.x;
            g[e + 1] = gsee * x.y;
          }
          if (refl > 0.0) {
            const float4 q = ld_shared_value<RES>(reinterpret_cast<const float4*>(
                fin + (size_t)(nv1 - 1 - (i0 + r)) * pitch + c0));
            const Vec<T> mirror = *reinterpret_cast<const Vec<T>*>(&q);
#pragma unroll
            for (int e = 0; e < VEC; e++) g[e] = fma(refl, (double)mirror.e[e], g[e]);
          }
#pragma unroll
          for (int e = 0; e < VEC; e++) xr[m][e] = (T)g[e];
        }
      }
    } else if (RES && !prime) {  // nothing flows in from the vacuum side
#pragma unroll
      for (int m = 0; m < M; m++)
#pragma unroll
        for (int e = 0; e < VEC; e++) xr[m][e] = (T)0;
    }
  };
  first_upwind();
  const T c2 = (T)p.c2;
  const T a2 = c2 < (T)0 ? -c2 : c2;
  // the source band in registers: the march's stores could alias Params
  const int band_lo = p.band_lo, band_hi = p.band_hi;
  const T* srcbase = sizeof(T) == 8 ? (const T*)a.tab.src : (const T*)a.tab.src32;

  const bool tail = s1 == nx;  // the march ends on the wall or the vacuum plane
  int it0 = 0;
  const int n_steps = RES ? rs.n_steps : 1;
  for (int step = 0; step < n_steps; step++) {
    if constexpr (RES) {
      if (step > 0) {
        unit_sync<NT>(bar);  // the producer has seen the new coefficients
        if (ctl[5]) return;
        InPtr x = fout;
        fout = const_cast<T*>(fin);
        fin = x;
        it0 += n_items;
        first_upwind();
      }
    }
    bool ok = true;
    for (int q = 0; q < n_items; q++) {
      const int st = (it0 + q) % NS;
      const bool compute = !(prime && q == 0);
      const int k = item_plane(q);
      // per-plane values are fetched before waiting for the stage, so their
      // latency overlaps the wait (RES: they come with the stage)
      // collision term (Eq. 3) of FP32 grids: dt nu_k and dt nu_k n_k (FP64
      // grids take it from the producer's row tables)
      float c1f = 0.f;
      T a1 = (T)0, bgk_a = (T)0, bgk_s = (T)0;
      if constexpr (!RES) {
        c1f = arg_at_use<SAU>(a.c1_32)[k];
        a1 = c1f == 0.f ? (T)0
                        : (sizeof(T) == 8 ? (T)fabs(arg_at_use<SAU>(a.c1)[k]) : (T)fabsf(c1f));
        if (BGK && sizeof(T) == 4) {
          const float* b32 = arg_at_use<SAU>(a.bgk32);
          bgk_a = (T)b32[k];
          bgk_s = (T)b32[nx + k];
        }
      }
      // source term: FP32 grids rebuild it from the separable factors in
      // shared memory, FP64 grids load the 2D table in the update loop
      const bool band = compute && k >= band_lo && k < band_hi;
      ok = !__any_sync(0xffffffffu,
                       !mbar_wait(&full[st], (uint32_t)(((it0 + q) / NS) & 1), wlim));
      if (!ok) {
        if (lane == 0) atomicOr(&a.st->flags, kFlagTimeout);
        if constexpr (!RES) return;
        if (lane == 0) ctl[4] = 1;
        break;
      }
      if constexpr (RES) {
        c1f = iv[st].c1;
        a1 = sizeof(T) == 8 ? (T)iv[st].a1 : (T)fabsf(c1f);
        if (BGK && sizeof(T) == 4) {
          bgk_a = (T)iv[st].bgk_a;
          bgk_s = (T)iv[st].bgk_s;
        }
      }
      // the tile's first row sits at stage row 1 when this plane's halo lies
      // above (c_1 > 0), at row 0 otherwise
      const int sbo = c1f > 0.f ? pitch : 0;  // sb's offset in the stage
      const T* sb = reinterpret_cast<const T*>(stage_base + st * sbytes) + sbo;
      if (!compute) {
#pragma unroll
        for (int m = 0; m < M; m++) {
          // (missing vectors' loads took thin FP64 batches 3 to 5 % longer: 64 grids of
          // 48-96 planes 154 -> 147 us a step)
          if (sizeof(T) == 8 && !(valid >> m & 1)) continue;
          if (!in_bounds(sbo + (int)(soff[m] & 0xFFFFFF) + VEC <= stage_n, a.st)) continue;
          const Vec<T> own = *reinterpret_cast<const Vec<T>*>(sb + (soff[m] & 0xFFFFFF));
#pragma unroll
          for (int e = 0; e < VEC; e++) xr[m][e] = own.e[e];
        }
      } else {
        // v1 upwind row: one row up (c_1 > 0), one down (c_1 < 0) or none;
        // the direction comes from the FP32 copy, as in the producer, so the
        // row read is always one that was copied or zero-filled
        const int nboff = c1f > 0.f ? -pitch : (c1f < 0.f ? pitch : 0);
        [[maybe_unused]] const double* dg = dgl + st * kMaxTileRows;
        T sum_n = (T)0;
        float sh_ = 0.f, sc_ = 0.f, sl_ = 0.f;  // FP64 grids: compensated FP32 sum
        T* oplane = (SAU ? static_cast<T*>(arg_at_use<SAU>(a.f_out)) : fout) + (size_t)k * plane;
        if constexpr (sizeof(T) == 4) {
          // FP32 grids, increment form: f' = f + (|c_2| (f_w - f) + (|c_1| (f_v - f)
          // + (|c_x| (f_x - f) + s))), two cells to an instruction.  No branch on a
          // thread's last, possibly missing vector: it computes the tile's first
          // cells again and neither stores nor sums them, which leaves the loads of
          // all vectors free to overlap.
          const F2 a1p = f2_pack(a1, a1), a2p = f2_pack(a2, a2);
          F2 sum2 = f2_pack(0.f, 0.f);
#pragma unroll
          for (int m = 0; m < M; m++) {
            if (NT * m >= rows * QV) break;  // no thread of the unit has vector m (uniform)
            const bool in = valid >> m & 1;
            const int so = soff[m] & 0xFFFFFF;
            const int r = soff[m] >> 24;
            float4 own = make_float4(0.f, 0.f, 0.f, 0.f), nb = own;
            if (in_bounds(sbo + so + VEC <= stage_n, a.st))
              own = *reinterpret_cast<const float4*>(sb + so);
            // v2 upwind (c_2 >= 0 since E_y <= 0): element j-1
            float left = __shfl_up_sync(0xffffffffu, own.w, 1);
            if (lane == 0 && !(zleft >> m & 1))
              left = in_bounds(sbo + so - 1 >= 0, a.st) ? sb[so - 1] : 0.f;
            if (zleft >> m & 1) left = 0.f;
            if (in_bounds(sbo + so + nboff >= 0 && sbo + so + nboff + VEC <= stage_n, a.st))
              nb = *reinterpret_cast<const float4*>(sb + so + nboff);
            const F2 f0 = f2_pack(own.x, own.y), f1 = f2_pack(own.z, own.w);
            F2 s0 = f2_pack(0.f, 0.f), s1 = s0;
            if (band) {  // separable source
              const float sr = srow_s[r];
              const float4 sc = *reinterpret_cast<const float4*>(scol_s + (so - r * pitch));
              s0 = f2_pack(sr * sc.x, sr * sc.y);
              s1 = f2_pack(sr * sc.z, sr * sc.w);
            }
            if (BGK) {  // dt nu_k n_k m1[i] m2[j] less the loss dt nu_k f
              const float ms = bgk_s * m1_s[r];
              const float4 mv = *reinterpret_cast<const float4*>(m2_s + (so - r * pitch));
              const F2 ms2 = f2_pack(ms, ms), ba2 = f2_pack(-bgk_a, -bgk_a);
              s0 = f2_fma(ba2, f0, f2_fma(ms2, f2_pack(mv.x, mv.y), s0));
              s1 = f2_fma(ba2, f1, f2_fma(ms2, f2_pack(mv.z, mv.w), s1));
            }
            const F2 axp = f2_pack(ax[m], ax[m]);
            s0 = f2_fma(axp, f2_sub(f2_pack(xr[m][0], xr[m][1]), f0), s0);
            s1 = f2_fma(axp, f2_sub(f2_pack(xr[m][2], xr[m][3]), f1), s1);
            s0 = f2_fma(a1p, f2_sub(f2_pack(nb.x, nb.y), f0), s0);
            s1 = f2_fma(a1p, f2_sub(f2_pack(nb.z, nb.w), f1), s1);
            s0 = f2_fma(a2p, f2_pack(left - own.x, own.x - own.y), s0);
            s1 = f2_fma(a2p, f2_pack(own.y - own.z, own.z - own.w), s1);
            F2 o0 = f2_add(f0, s0), o1 = f2_add(f1, s1);
            if (PADDED && (zleft >> (16 + m) & 1)) {  // row padding stays zero
              const int np = nv2 - (pitch - VEC);  // the vector's cells inside the grid
              float2 p0 = f2_unpack(o0), p1 = f2_unpack(o1);
              if (np <= 1) p0.y = 0.f;
              if (np <= 2) p1.x = 0.f;
              if (np <= 3) p1.y = 0.f;
              o0 = f2_pack(p0.x, p0.y);
              o1 = f2_pack(p1.x, p1.y);
            }
            // x-upwind value for the next plane is f^n here
            xr[m][0] = own.x;
            xr[m][1] = own.y;
            xr[m][2] = own.z;
            xr[m][3] = own.w;
            if (in) {
              sum2 = f2_add(sum2, f2_add(o0, o1));
              if (in_bounds((size_t)k * plane + gbase + so + VEC <= f_n, a.st)) {
                const float2 p0 = f2_unpack(o0), p1 = f2_unpack(o1);
                __stcs(reinterpret_cast<float4*>(oplane + so + gbase),
                       make_float4(p0.x, p0.y, p1.x, p1.y));
              }
            }
          }
          const float2 s2 = f2_unpack(sum2);
          sum_n = s2.x + s2.y;
        } else {
#pragma unroll
          for (int m = 0; m < M; m++) {
            if (NT * m >= rows * QV) break;  // no thread of the unit has vector m (uniform)
            const int so = soff[m] & 0xFFFFFF;
            Vec<T> own;
            if ((valid >> m & 1) && in_bounds(sbo + so + VEC <= stage_n, a.st))
              own = *reinterpret_cast<const Vec<T>*>(sb + so);
            else
#pragma unroll
              for (int e = 0; e < VEC; e++) own.e[e] = (T)0;
            // v2 upwind (c_2 >= 0 since E_y <= 0): element j-1
            T left = __shfl_up_sync(0xffffffffu, own.e[VEC - 1], 1);
            if (!(valid >> m & 1)) continue;
            if (zleft >> m & 1)
              left = (T)0;
            else if (lane == 0)
              left = in_bounds(sbo + so - 1 >= 0, a.st) ? sb[so - 1] : (T)0;
            Vec<T> nb;
            if (in_bounds(sbo + so + nboff >= 0 && sbo + so + nboff + VEC <= stage_n, a.st))
              nb = *reinterpret_cast<const Vec<T>*>(sb + so + nboff);
            else
#pragma unroll
              for (int e = 0; e < VEC; e++) nb.e[e] = (T)0;
            const T d = dg[soff[m] >> 24];
            Vec<T> src;
#pragma unroll
            for (int e = 0; e < VEC; e++) src.e[e] = (T)0;
            if (band) src = *reinterpret_cast<const Vec<T>*>(srcbase + so + gbase);
            if (BGK) {  // gain dt nu_k n_k m1[i] m2[j] of the collision term
              const int r = soff[m] >> 24;
              const int c0 = so - r * pitch;  // column of the vector's first cell
              const double ms = dgs[st * kMaxTileRows + r];
              const Vec<double> mv = *reinterpret_cast<const Vec<double>*>(m2d + c0);
#pragma unroll
              for (int e = 0; e < VEC; e++) src.e[e] = fma(ms, mv.e[e], src.e[e]);
            }
            Vec<T> out;
#pragma unroll
            for (int e = 0; e < VEC; e++) {
              const T f = own.e[e];
              const T fw = e == 0 ? left : own.e[e - 1];
              T fn = upd(f, xr[m][e], nb.e[e], fw, ax[m], a1, a2, src.e[e], d);
              if (PADDED && (zleft >> (16 + m) & 1) && e >= nv2 - (pitch - VEC))
                fn = (T)0;  // row padding stays zero
              out.e[e] = fn;
              xr[m][e] = f;  // x-upwind value for the next plane is f^n here
              float h, l;
              split_double((double)fn, h, l);
              two_sum_acc(sh_, sc_, h);
              sl_ += l;
            }
            if (in_bounds((size_t)k * plane + gbase + so + VEC <= f_n, a.st))
              __stcs(reinterpret_cast<float4*>(oplane + so + gbase),
                     *reinterpret_cast<const float4*>(&out));
          }
        }
        // warp sum of this plane's f^{n+1} (an FP32 grid sums its 32 lanes in
        // FP32; everything above a warp is FP64)
        double* wsl = wsum + (st * kWarps + warp) * kWs;
        if (sizeof(T) == 4) {
          const T ws = warp_sum(sum_n);
          if (lane == 0) *reinterpret_cast<float*>(wsl) = ws;  // the producer converts once
        } else {
          // fold the lanes' (hi, error) pairs in FP32 with TwoSum; the producer
          // converts them
          float lo = sc_ + sl_;
          for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_down_sync(0xffffffffu, sh_, o);
            const float ol = __shfl_down_sync(0xffffffffu, lo, o);
            float c = 0.f;
            two_sum_acc(sh_, c, oh);
            lo += ol + c;
          }
          if (lane == 0) *reinterpret_cast<float2*>(wsl) = make_float2(sh_, lo);
        }
        const bool wall = !RES && k == 0 && dir < 0, vout = !RES && k == nx - 1 && dir > 0;
        if (wall || vout) {  // uniform over the block
          double b3[3];
          if constexpr (sizeof(T) == 4 && NT == kHalfThreads) {
            const bool neg = wall_terms_pairs(oplane, a.tab.v1p, a.tab.deltap, tid, NT, i0, rows,
                                              nv2, pitch, wall, b3);
            if (__any_sync(0xffffffffu, neg) && lane == 0) atomicOr(&a.st->flags, kFlagNegative);
            if (lane == 0) {
              wsl[1] = b3[0];
              wsl[2] = b3[1];
              wsl[3] = b3[2];
            }
          } else {
            const bool neg =
                wall_terms<T>(oplane, a.tab.v1, a.tab.vdelta, tid, NT, i0, rows, nv2, pitch, wall, b3);
            if (__any_sync(0xffffffffu, neg) && lane == 0) atomicOr(&a.st->flags, kFlagNegative);
            const double w1 = warp_sum(b3[0]), w2 = warp_sum(b3[1]), w3 = warp_sum(b3[2]);
            if (lane == 0) {
              wsl[1] = w1;
              wsl[2] = w2;
              wsl[3] = w3;
            }
          }
        } else if (k == 0 || k == nx - 1) {
          if (lane == 0) wsl[1] = wsl[2] = wsl[3] = 0.0;
        }
      }
      if (RES && tail && q == n_items - 1) continue;  // its boundary sums follow
      mbar_arrive(&empty[st]);  // this thread is done with stage st
    }
    if constexpr (RES) {
      if (tail && ok) {
        // the boundary plane's sums: what was stored is read back
        const int st = (it0 + n_items - 1) % NS;
        const int k = item_plane(n_items - 1);
        double* wsl = wsum + (st * kWarps + warp) * kWs;
        double b3[3];
        const bool neg = wall_terms_ahead<T, sizeof(T) == 4 && NT == kHalfThreads>(
            fout + (size_t)k * plane, a.tab, tid, NT, i0, rows, pitch, dir < 0, b3);
        if (__any_sync(0xffffffffu, neg) && lane == 0) atomicOr(&a.st->flags, kFlagNegative);
        if (lane == 0) {
          wsl[1] = b3[0];
          wsl[2] = b3[1];
          wsl[3] = b3[2];
        }
        __syncwarp();
        mbar_arrive(&empty[st]);
      }
      end_step();
      if (ctl[4]) return;
    }
  }
}

// Shared memory of one unit: argument slot, stages and tail.  A CTA of two
// half units holds two such regions, each rounded up to 128 bytes.
template <typename T, int NS>
__host__ __device__ constexpr size_t unit_smem_bytes(int stage_elems, int pitch) {
  return NS * stage_bytes<T>(stage_elems) + tail_bytes<T, NS>(pitch);
}
template <typename T>
__host__ __device__ constexpr size_t half_region_bytes(int stage_elems, int pitch) {
  return (unit_smem_bytes<T, kHalfStages>(stage_elems, pitch) + 127) / 128 * 128;
}

}  // namespace
}  // namespace fk
