// The finalize step (moments -> surface charge, field, Courant numbers,
// ledger, history) as device code shared by the finalize kernels and the
// resident step kernel, and the block reductions it uses.
//
// Paper: Sun et al., arXiv 2303.14119, Sec. 2.
#pragma once

#include <math.h>

#include "fk_host.cuh"

namespace fk {
namespace {

// ---------------------------------------------------------------------------
// Deterministic block reductions: fixed shuffle tree, fixed warp order.
template <int NT>
__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    r = l < NT / 32 ? sh[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;  // valid in thread 0
}

template <int NT>
__device__ __forceinline__ double block_max(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    r = l < NT / 32 ? sh[l] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r = fmax(r, __shfl_down_sync(0xffffffffu, r, o));
  }
  return r;
}

// ---------------------------------------------------------------------------
// Finalize, after every step kernel (and after a moments-only evaluation).
//
// Phase A, one thread per x-plane over kFinBlocks-sized blocks: the plane's
// density n_k from its tile partials (fixed order), the velocity-edge loss,
// and the exclusive prefix of n within the block.  Phase B, run by the last
// block to finish (a counter in FinScratch decides which; its sums are in a
// fixed order, so the result does not depend on which block it is):
//  - step mode: ledger += dt * (fluxes of f^n), sigma^{n+1} = sigma^n +
//    e dt (Gamma_see^n - Gamma_pe^n)  (Eq. 18 summed with Eq. 14), step++;
//    in the Strang step mode the wall and vacuum terms of f^n weigh dt/2
//    (the other half was added after the velocity pass);
//  - the fluxes of the new state (Eqs. 12-14), N, and the history row;
//  - E_x from Gauss's law integrated from the wall, E_x(0) = sigma/(2 eps0)
//    (the Poisson problem of Sec. 2), c_1 = -e E_x dt / (m_e dv1);
//  - CFL and finiteness checks (sticky flags) and the convergence test
//    (Sec. 2, paragraph after Eq. 18).
// Spreading phase A over many SMs matters on GB300, whose FP64 rate per SM
// is a small fraction of its FP32 rate.
constexpr int kFinThreads = 128;
constexpr int kFinMaxBlocks = 64;  // nx <= 8192

// E_x at the centre of a plane of density n_k with `below` the densities
// between the wall and it (Gauss's law).
__device__ __forceinline__ double field_at(double e_wall, double ex_n, double below, double n_k) {
  return fma(-ex_n, fma(0.5, n_k, below), e_wall);
}
// sigma^{n+1} from the fluxes of f^n (Eq. 18); hw: the wall terms' share of dt.
__device__ __forceinline__ double advance_sigma(double sigma, double hw, double g_see, double g_pe,
                                                double refl) {
  return fma(kQe * hw, fma(-(1.0 - refl), g_pe, g_see), sigma);
}
// The ledger's share of one step with the fluxes of f^n in d and the
// velocity-edge loss l; the step count.
__device__ __forceinline__ void advance_ledger(DevState& d, const Params& p, double l, double hw) {
  d.cum_emit = fma(hw, fma(p.refl, d.g_pe, d.g_see), d.cum_emit);  // secondaries and reflected
  d.cum_see = fma(hw, d.g_see, d.cum_see);
  d.cum_pe = fma(hw, d.g_pe, d.cum_pe);
  d.cum_vac = fma(hw, d.g_vac, d.cum_vac);
  d.cum_lv = fma(p.dt, l * p.lv_scale, d.cum_lv);
  d.cum_inj = fma(p.dt, p.inj, d.cum_inj);
  d.step += 1;
}
// The history row of the new state in d, and (stepping) the convergence test
// against the row a window before it.
__device__ __forceinline__ void append_history(DevState& d, const Params& p, double* hist,
                                               double ex0, bool stepping) {
  const long long row = d.step, cap = p.hist_cap, window = p.sat_window;
  const double rr[FK_HISTORY_COLS] = {(double)row, (double)row * p.dt, d.sigma, d.g_pe,
                                      d.g_see, d.g_vac, d.n_tot, ex0};
  double* r = hist + (size_t)(row % cap) * FK_HISTORY_COLS;
  for (int q = 0; q < FK_HISTORY_COLS; q++) r[q] = rr[q];
  if (row + 1 > d.hist_count) d.hist_count = row + 1;
  if (stepping && d.sat_step < 0 && row >= window && window < cap) {
    const double* o = hist + (size_t)((row - window) % cap) * FK_HISTORY_COLS;
    bool ok = true;
    for (int q = 2; q <= 4; q++)
      if (!(fabs(rr[q] - __ldcg(o + q)) <= p.sat_tol * fabs(rr[q]))) ok = false;
    if (ok) d.sat_step = row;
  }
}

// Block blk of nblk finalizing one grid.
__device__ __forceinline__ void finalize_body(const StepArgs& a, const FinOut& o, const int blk,
                                              const int nblk, const int mode) {
  double* const ne = o.ne;
  double* const Ex = o.Ex;
  double* const c1 = o.c1;
  float* const c1_32 = o.c1_32;
  double* const hist = o.hist;
  const FinScratch& fs = o.fs;
  __shared__ double sh[32];
  __shared__ double wscan[kFinThreads / 32];
  __shared__ int s_last;
  __shared__ double bc[4];
  __shared__ double boff[kFinMaxBlocks];  // phase B: sum of n over blocks below
  const Params& p = *a.prm;
  DevState* st = a.st;
  const bool stepping = mode == kModeStep || mode == kModeStepStrang;
  if (stepping && st->flags) return;
  const int nx = a.nx, nu = a.part.nu;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int k = blk * kFinThreads + t;
  // ---- phase A
  double nk = 0.0, lk = 0.0;
  if (k < nx) {
    // loads batched ahead of the (fixed-order) adds: in-order issue would
    // otherwise serialise one L2 round trip per partial
    const double* pn = a.part.n + (size_t)k * nu;
    const double* pl = a.part.lv + (size_t)k * nu;
    double sn = 0.0, sl = 0.0;
    int u = 0;
    for (; u + 8 <= nu; u += 8) {
      double xn[8], xl[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        xn[q] = pn[u + q];
        xl[q] = pl[u + q];
      }
#pragma unroll
      for (int q = 0; q < 8; q++) {
        sn += xn[q];
        sl += xl[q];
      }
    }
    for (; u < nu; u++) {
      sn += pn[u];
      sl += pl[u];
    }
    nk = sn * p.dvv;
    lk = sl;
    ne[k] = nk;
  }
  double incl = nk;
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  double excl = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) excl = 0.0;
  if (lane == 31) wscan[w] = incl;
  __syncthreads();
  double woff = 0.0;
  for (int q = 0; q < w; q++) woff += wscan[q];
  if (k < nx) fs.pre[k] = woff + excl;  // sum of n over the block's planes below k
  const double blv = block_sum<kFinThreads>(lk, sh);
  if (t == 0) {
    double btot = 0.0;  // the scan's own end: no second sum over the planes
    for (int q = 0; q < kFinThreads / 32; q++) btot += wscan[q];
    fs.bsum[blk] = btot;
    fs.blv[blk] = blv;
    __threadfence();
    s_last = atomicAdd(fs.counter, 1) == nblk - 1;
  }
  __syncthreads();
  if (!s_last) return;
  // ---- phase B (last block)
  __threadfence();
  const int nb = nblk;
  if (w == 0) {
    // block totals and their exclusive prefix, wall-flux tile partials:
    // lane-strided loads, fixed shuffle trees (other blocks' results are
    // read past L1 with __ldcg)
    const double b0 = lane < nb ? __ldcg(fs.bsum + lane) : 0.0;
    const double b1 = lane + 32 < nb ? __ldcg(fs.bsum + lane + 32) : 0.0;
    double l = (lane < nb ? __ldcg(fs.blv + lane) : 0.0) +
               (lane + 32 < nb ? __ldcg(fs.blv + lane + 32) : 0.0);
    double i0s = b0, i1s = b1;  // inclusive scans of the two halves
    for (int o = 1; o < 32; o <<= 1) {
      const double y0 = __shfl_up_sync(0xffffffffu, i0s, o);
      const double y1 = __shfl_up_sync(0xffffffffu, i1s, o);
      if (lane >= o) {
        i0s += y0;
        i1s += y1;
      }
    }
    // the totals where the blocks end
    const double half = __shfl_sync(0xffffffffu, i0s, min(nb, 32) - 1);
    if (lane < nb) boff[lane] = i0s - b0;
    if (lane + 32 < nb) boff[lane + 32] = half + i1s - b1;
    const double ntot_raw = nb > 32 ? half + __shfl_sync(0xffffffffu, i1s, nb - 33) : half;
    double pe = 0.0, see = 0.0, vac = 0.0;
    for (int u = lane; u < nu; u += 32) {
      pe += a.part.pe[u];
      see += a.part.see[u];
      vac += a.part.vac[u];
    }
    for (int o = 16; o > 0; o >>= 1) {
      l += __shfl_down_sync(0xffffffffu, l, o);
      pe += __shfl_down_sync(0xffffffffu, pe, o);
      see += __shfl_down_sync(0xffffffffu, see, o);
      vac += __shfl_down_sync(0xffffffffu, vac, o);
    }
    if (lane == 0) {
      *fs.counter = 0;  // ready for the next launch
      DevState d = *st;  // one batch of loads, updated in registers
      const double ntot = ntot_raw * p.dx;
      pe *= p.dvv;
      // secondaries come from the absorbed part (1 - refl) of the primaries;
      // with SEE off every absorbed primary is deposited
      see = p.see_enabled ? see * p.dvv * (1.0 - p.refl) : 0.0;
      vac *= p.dvv;
      if (stepping) {
        const double hw = mode == kModeStepStrang ? 0.5 * p.dt : p.dt;  // wall terms' share
        d.sigma = advance_sigma(d.sigma, hw, d.g_see, d.g_pe, p.refl);
        advance_ledger(d, p, l, hw);
      }
      if (mode == kModeReset) {
        d.step = 0;
        d.hist_count = 0;
        d.sat_step = -1;
        d.cum_emit = d.cum_see = d.cum_pe = d.cum_vac = d.cum_lv = d.cum_inj = 0.0;
        d.sigma0 = d.sigma;
        d.n0 = ntot;
      }
      d.g_pe = pe;
      d.g_see = see;
      d.g_vac = vac;
      d.n_tot = ntot;
      if (!isfinite(pe) || !isfinite(see) || !isfinite(vac) || !isfinite(ntot) ||
          !isfinite(d.sigma))
        d.flags |= kFlagNumeric;
      *st = d;  // one batch of stores
      bc[0] = d.sigma;
    }
  }
  __syncthreads();
  const double e_wall = bc[0] * p.ex_sigma;
  // E_x at cell centres and the v1-Courant numbers.  The planes' prefix
  // sums and densities (other blocks' results) are loaded kLd at a time, and
  // the coefficients once, ahead of the stores, past which the compiler
  // cannot move a load.
  const bool self_cons = p.self_consistent, coll = p.collisions;
  const double ex_n = p.ex_n, ex_ext = p.Ex_ext, c1_per_ex = p.c1_per_ex, bgk_c = p.bgk_c;
  const double cx_max = p.cx_max, ac2 = fabs(p.c2);
  double cmax = 0.0, ex0 = 0.0;
  constexpr int kLd = 8;
  for (int k0 = t; k0 < nx; k0 += kLd * kFinThreads) {
    double pre_l[kLd], ne_l[kLd];
#pragma unroll
    for (int j = 0; j < kLd; j++) {
      const int kk = k0 + j * kFinThreads;
      pre_l[j] = kk < nx ? __ldcg(fs.pre + kk) : 0.0;
      ne_l[j] = kk < nx ? __ldcg(ne + kk) : 0.0;
    }
#pragma unroll
    for (int j = 0; j < kLd; j++) {
      const int kk = k0 + j * kFinThreads;
      if (kk >= nx) break;
      const double below = boff[kk / kFinThreads] + pre_l[j];
      const double n_k = ne_l[j];
      const double e = self_cons ? field_at(e_wall, ex_n, below, n_k) : ex_ext;
      if (kk == 0) ex0 = e;
      Ex[kk] = e;
      const double c = c1_per_ex * e;
      c1[kk] = c;
      c1_32[kk] = (float)c;
      double cfl = fabs(c);
      if (coll) {
        // BGK coefficients of the new state (Eqs. 3-4): dt nu_k = bgk_c n_k
        const double ak = n_k > 0.0 ? bgk_c * n_k : 0.0;
        a.bgk[kk] = ak;
        a.bgk[nx + kk] = ak * n_k;
        a.bgk32[kk] = (float)ak;
        a.bgk32[nx + kk] = (float)(ak * n_k);
        cfl += ak;  // the collision term takes part in the positivity bound
      }
      cmax = fmax(cmax, cfl);
    }
  }
  cmax = block_max<kFinThreads>(cmax, sh);
  __syncthreads();
  if (t == 0) {
    DevState d = *st;
    if (cmax + cx_max + ac2 > 1.0 + 1e-12) d.flags |= kFlagCfl;
    append_history(d, p, hist, ex0, stepping);
    st->flags = d.flags;
    st->hist_count = d.hist_count;
    st->sat_step = d.sat_step;
  }
}

}  // namespace
}  // namespace fk
