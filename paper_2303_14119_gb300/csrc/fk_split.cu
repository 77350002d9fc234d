// Split time steps (Lie and Strang) in one march over f.
//
// The split step as passes of the streaming kernel moved f once per pass
// (Lie: two reads and two writes, Strang: three of each, and a launch for
// each).  The velocity step takes its coefficients from f^n, so nothing
// global stands between the passes but the wall fluxes of the state after the
// velocity step, which enter only the x = 0 plane of the rows with v1 > 0.
// One march therefore does the whole step:
//
//   g  = x-step of f^n (dt, or dt/2 for Strang)   own rows and one halo row
//   h  = velocity step of g                       (v1, v2, source, collisions)
//   f' = h (Lie) or the x-step of h over dt/2 (Strang)
//
// and a small kernel completes the x = 0 plane of a Strang step.
//
// Measured, us a step, passes -> here: Strang 512 x 128 x 128 FP32 66 -> 44,
// FP64 270 -> 164, 1024 x 256 x 256 FP32 309 -> 162, 64 x 48 x 48 FP64 85 ->
// 37; Lie 1024 x 256 x 256 FP32 207 -> 118, 512 x 256 x 256 FP64 623 -> 429.
// Small grids are bound by the launches and the finalize, FP64 grids by the
// FP64 pipe (5 operations a cell for Lie and 7 for Strang, where the passes
// took 8 and 12), large FP32 ones by the latency of a plane's two phases.
//
// Decomposition: as the streaming kernel's, a CTA owns (tile of v1 rows of one
// sign, chunk of planes) and marches with the x-upwind direction; a thread
// keeps the previous plane's f and h of its cells in registers.  The one or
// two planes upwind of the chunk are computed again.  A stage of shared
// memory holds a plane's rows of the tile, the v1 halo row on the upwind side
// of that plane's c_1, and that halo row's own x-upwind neighbour (its sign of
// v1 can differ from the tile's).  g replaces f in the stage; after the one
// barrier of a plane every thread reads its neighbours there.  That barrier
// also frees the stage before it, which thread 0 refills by bulk copies: two
// planes in flight for each CTA, two or three CTAs on an SM.
//
// Paper: Sun et al., arXiv 2303.14119, Sec. 2 (the update of Eq. 2; splitting
// is this library's).
#include <algorithm>

#include "fk_host.cuh"
#include "fk_split.cuh"
#include "fk_stream_unit.cuh"

namespace fk {

namespace {

constexpr int kSplitThreads = 256;
constexpr int kSplitWarps = kSplitThreads / 32;
constexpr int kSplitStages = 3;     // 4: the same, or slower where a CTA less fits an SM
constexpr int kSplitVec = 4;        // 16-byte vectors per thread and plane
// planes of a chunk, at least: with 1 instead of 2 a 64 x 48 x 48 FP64 Lie step
// took 19 us instead of 25 (each plane is a chain of two phases)
constexpr int kSplitMinChunk = 1;
// planes that the boundary sums of a march's last plane are worth
constexpr int kSplitLast = 2;

// Shared memory after the stages.
struct SplitShared {
  uint64_t full[kSplitStages];
  float2 wn[2][kSplitWarps];        // a plane's warp sums (and their errors)
  double wall[2][kSplitWarps][3];                  // boundary sums of h and f'
};
template <typename T>
__host__ __device__ constexpr size_t split_tail_bytes(int pitch) {
  // row and column factors: source and collisions
  return sizeof(SplitShared) + 2 * ((size_t)kMaxTileRows + pitch) * sizeof(T) + 16;
}
template <typename T>
__host__ __device__ constexpr size_t split_smem_bytes(int stage_elems, int pitch) {
  return kSplitStages * stage_bytes<T>(stage_elems) + split_tail_bytes<T>(pitch);
}

// x-step of one cell, in the streaming kernel's arithmetic: convex form of
// FP64 grids (d = 1 - ax), increment form of FP32 grids.
__device__ __forceinline__ double x_step(double f, double fx, double ax, double d) {
  return fma(ax, fx, d * f);
}
__device__ __forceinline__ float x_step(float f, float fx, float ax, float) {
  return __fadd_rn(f, __fmul_rn(ax, fx - f));
}
__device__ __forceinline__ Vec<double> x_step_vec(const Vec<double>& f, const double (&fx)[2], double ax,
                                                  double d) {
  return Vec<double>{{x_step(f.e[0], fx[0], ax, d), x_step(f.e[1], fx[1], ax, d)}};
}
__device__ __forceinline__ Vec<float> x_step_vec(const Vec<float>& f, const float (&fx)[4], float ax,
                                                 float) {
  const F2 f0 = f2_pack(f.e[0], f.e[1]), f1 = f2_pack(f.e[2], f.e[3]), a2 = f2_pack(ax, ax);
  const float2 r0 = f2_unpack(f2_add(f0, f2_mul(a2, f2_sub(f2_pack(fx[0], fx[1]), f0))));
  const float2 r1 = f2_unpack(f2_add(f1, f2_mul(a2, f2_sub(f2_pack(fx[2], fx[3]), f1))));
  return Vec<float>{{r0.x, r0.y, r1.x, r1.y}};
}

// CTAs on an SM: a Lie step of FP32 grids holds half the registers of a Strang
// step (three: 118 us at 1024 x 256 x 256, two: 136); three of a Strang step
// spill (two: 163 us, three: 211), and FP64 grids are bound by their pipe.
template <typename T, bool STRANG, bool BGK>
__global__ void __launch_bounds__(kSplitThreads, sizeof(T) == 4 && !STRANG ? 3 : 2)
split_kernel(const __grid_constant__ SplitArgs sa) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int NT = kSplitThreads, NW = kSplitWarps, NS = kSplitStages, M = kSplitVec;
  constexpr int VEC = Vec<T>::N;
  constexpr int D = STRANG ? 2 : 1;  // planes upwind of a chunk that it needs
  const StepArgs& a = sa.a;
  const Geom& gm = a.geom;
  const Params& p = *a.prm;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nx = a.nx, nv1 = a.nv1, nv2 = a.nv2, pitch = a.pitch, nt = gm.n_tiles;
  const int t = blockIdx.x % nt, chunk = blockIdx.x / nt;
  int i0, i1, dir;
  tile_rows(gm, nv1, t, &i0, &i1, &dir);
  const int s0 = chunk * gm.chunk_len, s1 = min(nx, s0 + gm.chunk_len);
  if (s0 >= s1 || i0 >= i1) return;
  const int rows = i1 - i0, QV = pitch / VEC, nvec = rows * QV;
  const size_t plane = (size_t)nv1 * pitch;
  if (!in_bounds(rows <= kMaxTileRows && (rows + 3) * pitch <= gm.stage_elems && nvec <= NT * M, a.st))
    return;
  const size_t sbytes = stage_bytes<T>(gm.stage_elems);
  SplitShared& sh = *reinterpret_cast<SplitShared*>(smem + NS * sbytes);
  // FP32: source factors of the rows, FP64: 1 - |c_x| (or half); both: collision factors
  T* const srow = reinterpret_cast<T*>(&sh + 1);
  T* const m1 = srow + kMaxTileRows;
  T* const scol = reinterpret_cast<T*>((reinterpret_cast<uintptr_t>(m1 + kMaxTileRows) + 15) & ~(uintptr_t)15);
  T* const m2 = scol + pitch;
  for (int r = tid; r < rows; r += NT) {
    srow[r] = sizeof(T) == 4 ? (T)a.tab.srow32[i0 + r]
                             : (T)(1.0 - (STRANG ? 0.5 : 1.0) * fabs(a.tab.cx[i0 + r]));
    if (BGK) m1[r] = sizeof(T) == 8 ? (T)a.tab.m1[i0 + r] : (T)a.tab.m1_32[i0 + r];
  }
  for (int j = tid; j < pitch; j += NT) {
    if (sizeof(T) == 4) scol[j] = (T)a.tab.scol32[j];
    if (BGK) m2[j] = sizeof(T) == 8 ? (T)a.tab.m2[j] : (T)a.tab.m2_32[j];
  }
  if (tid == 0) {
    for (int s = 0; s < NS; s++) mbar_init(&sh.full[s], 1);
    fence_mbar_init();
  }
  if (__syncthreads_or(tid == 0 && *const_cast<volatile unsigned*>(&a.st->flags) != 0))
    return;  // sticky error: freeze the state

  const T* const fin = static_cast<const T*>(a.f_in);
  T* const fout = static_cast<T*>(a.f_out);
  const long long* const wlim = &p.wait_limit;
  const double gsee = a.st->g_see, refl = p.refl;

  // items of the march: step s visits plane s or nx - 1 - s; the first one
  // only primes the x-upwind values unless the march begins at the boundary
  const int s_first = max(0, s0 - D);
  const bool raw = s0 >= D;
  const int n_items = s1 - s_first;
  auto plane_of = [&](int q) { return dir > 0 ? s_first + q : nx - 1 - (s_first + q); };
  // the halo row for a c_1 (-1: none inside the grid)
  auto halo_row = [&](float c1) {
    return c1 > 0.f ? i0 - 1 : (c1 < 0.f ? (i1 < nv1 ? i1 : -1) : -1);
  };
  const int withheld = (t == 0 && chunk == 0) ? p.withhold_item : -1;
  // thread 0: copy item q, whose plane has the v1-Courant number c1
  auto issue = [&](int q, float c1) {
    if (q == withheld) return;  // test knob
    const int k = plane_of(q), st = q % NS;
    T* stage = reinterpret_cast<T*>(smem + st * sbytes);
    const int ih = raw && q == 0 ? -1 : halo_row(c1);
    int lo = i0, n = rows;
    if (ih >= 0) {
      n++;
      if (ih < i0) lo = ih;
    }
    int ku = -1;  // the halo row's x-upwind plane
    if (ih >= 0) ku = ih < gm.i_neg ? k + 1 : k - 1;
    const bool up = ih >= 0 && ku >= 0 && ku < nx;
    const uint32_t row = (uint32_t)(pitch * (int)sizeof(T));
    if (!in_bounds(k >= 0 && k < nx && lo >= 0 && lo + n <= nv1, a.st)) {
      mbar_expect_tx(&sh.full[st], 0);
      return;
    }
    mbar_expect_tx(&sh.full[st], row * (uint32_t)(n + (up ? 1 : 0)));
    bulk_g2s(stage + (lo - i0 + 1) * pitch, fin + (size_t)k * plane + (size_t)lo * pitch, row * n,
             &sh.full[st]);
    if (up)
      bulk_g2s(stage + (rows + 2) * pitch, fin + (size_t)ku * plane + (size_t)ih * pitch, row,
               &sh.full[st]);
  };
  float c1_issue = 0.f;  // thread 0: c_1 of the next item to be copied
  if (tid == 0) {
    for (int q = 0; q < min(NS, n_items); q++) issue(q, a.c1_32[plane_of(q)]);
    if (n_items > NS) c1_issue = a.c1_32[plane_of(NS)];
  }

  // this thread's vectors: vector m is the tile's vector tid + NT m, at the
  // same offset in a stage's rows and in the plane's; rws holds their rows (a
  // byte each), flg bit m: vector m exists, 8 + m: it starts a row (or does
  // not exist), 16 + m: it holds column nv2 - 1
  auto abs_cx = [&](int i) {
    const T cx = sizeof(T) == 8 ? (T)a.tab.cx[i] : (T)a.tab.cx32[i];
    return (STRANG ? (T)0.5 : (T)1) * (cx < (T)0 ? -cx : cx);
  };
  const int so0 = tid * VEC;
  unsigned flg = 0, rws = 0;
  static_assert(M <= 4 && kMaxTileRows <= 256, "a byte for each row");
  T ax[M], xr[M][VEC], hr[M][VEC];
#pragma unroll
  for (int m = 0; m < M; m++) {
    const int v = tid + NT * m;
    ax[m] = (T)0;
#pragma unroll
    for (int e = 0; e < VEC; e++) xr[m][e] = hr[m][e] = (T)0;
    if (v >= nvec || !in_bounds((v + 1) * VEC + 2 * pitch <= gm.stage_elems &&
                                    (size_t)i0 * pitch + (size_t)(v + 1) * VEC <= plane,
                                a.st)) {
      flg |= 256u << m;
    } else {
      const int r = v / QV, qv = v - r * QV;
      flg |= 1u << m;
      if (qv == 0) flg |= 256u << m;
      if (qv == QV - 1) flg |= 65536u << m;
      rws |= (unsigned)r << (8 * m);
      ax[m] = abs_cx(i0 + r);
    }
  }
  // a vector past the tile reads a vector of the halo row's place and drops
  // it: no branch stands before the loads of the others
  auto offset = [&](int m) { return flg >> m & 1 ? so0 + NT * VEC * m : -VEC; };
  const T ax_above = i0 > 0 ? abs_cx(i0 - 1) : (T)0, ax_below = i1 < nv1 ? abs_cx(i1) : (T)0;
  auto row_of = [&](int m) { return (int)(rws >> (8 * m) & 0xFF); };
  // the inflow at the wall into row i (v1 > 0), columns c .. c + VEC - 1: the
  // re-emitted distribution of Eq. 15 and the reflected part of f^n
  auto wall_inflow = [&](int i, int c) {
    Vec<T> out;
#pragma unroll
    for (int e = 0; e < VEC; e++) {
      double g = gsee * a.tab.gse[(size_t)i * pitch + c + e];
      if (refl > 0.0) g = fma(refl, (double)fin[(size_t)(nv1 - 1 - i) * pitch + c + e], g);
      out.e[e] = (T)g;
    }
    return out;
  };
  if (s_first == 0 && !raw && dir > 0) {
#pragma unroll
    for (int m = 0; m < M; m++)
      if (flg >> m & 1) {
        const int r = row_of(m);
        const Vec<T> w = wall_inflow(i0 + r, so0 + NT * VEC * m - r * pitch);
#pragma unroll
        for (int e = 0; e < VEC; e++) xr[m][e] = w.e[e];
      }
  }
  const T a2 = (T)fabs(p.c2);
  const bool has_a2 = p.c2 != 0.0;
  const double d2 = 1.0 - fabs(p.c2);
  const int band_lo = p.band_lo, band_hi = p.band_hi;
  const bool padded = nv2 != pitch;
  const int last_e = (nv2 - 1) % VEC;  // column nv2 - 1 in the last vector of a row

  // a plane's coefficients, fetched one plane ahead (and not touched before)
  struct Coef {
    float c1;
    T v1, ba, bs;  // v1: c_1 of an FP64 grid
  };
  auto load_coef = [&](int q) {
    Coef c{0.f, (T)0, (T)0, (T)0};
    if (q >= n_items) return c;
    const int k = plane_of(q);
    c.c1 = a.c1_32[k];
    if (sizeof(T) == 8) c.v1 = (T)a.c1[k];
    if (BGK) {
      c.ba = sizeof(T) == 8 ? (T)a.bgk[k] : (T)a.bgk32[k];
      c.bs = sizeof(T) == 8 ? (T)a.bgk[nx + k] : (T)a.bgk32[nx + k];
    }
    return c;
  };
  // FP64 instructions take 16 cycles of the SM whether one lane needs them or
  // 32: the sums above a thread are one warp's work.
  // one warp: fold the warps' sums of plane k (slot b) and store them
  auto fold = [&](int k, int b) {
    const float2 x = sh.wn[b][lane % NW];
    double n = sizeof(T) == 4 ? (double)x.x : (double)x.x + (double)x.y;
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1) n += __shfl_down_sync(0xffffffffu, n, o);
    if (lane == 0) a.part.n[(size_t)k * nt + t] = n;
  };
  // one warp: the outflow of g (plane k, in the stage at sb) through the
  // downwind velocity edges, for the ledger
  auto edge_loss = [&](int k, const T* sb, int erow, T a1) {
    T lv = (T)0;
    if (erow >= 0) {
      for (int j = lane; j < nv2; j += 32) lv += sb[erow * pitch + j];
      lv *= a1;
    }
    if (has_a2) {
      T x = (T)0;
      for (int r = lane; r < rows; r += 32) x += sb[r * pitch + nv2 - 1];
      lv += a2 * x;
    }
    lv = warp_sum(lv);
    if (lane == 0) a.part.lv[(size_t)k * nt + t] = (double)lv;
  };

  Coef next = load_coef(0);
  bool ok = true;
  int q = 0;
  for (; q < n_items; q++) {
    const int st = q % NS, k = plane_of(q);
    const Coef co = next;
    next = load_coef(q + 1);
    const T a1 = co.c1 == 0.f ? (T)0 : (sizeof(T) == 8 ? (T)fabs(co.v1) : (T)fabsf(co.c1));
    T* const stage = reinterpret_cast<T*>(smem + st * sbytes);
    T* const sb = stage + pitch;  // the tile's first row
    ok = mbar_wait(&sh.full[st], (uint32_t)((q / NS) & 1), wlim);
    const bool prime = raw && q == 0;
    // ---- x-step of f^n, in place
    if (prime) {
#pragma unroll
      for (int m = 0; m < M; m++) {
        if (NT * m >= nvec) break;
        const Vec<T> own = *reinterpret_cast<const Vec<T>*>(sb + offset(m));
#pragma unroll
        for (int e = 0; e < VEC; e++) xr[m][e] = own.e[e];
      }
    } else if (ok) {
#pragma unroll
      for (int m = 0; m < M; m++) {
        if (NT * m >= nvec) break;
        T* const c = sb + offset(m);
        const Vec<T> own = *reinterpret_cast<const Vec<T>*>(c);
        const Vec<T> g = x_step_vec(own, xr[m], ax[m], sizeof(T) == 8 ? srow[row_of(m)] : (T)0);
        if (flg >> m & 1) *reinterpret_cast<Vec<T>*>(c) = g;
#pragma unroll
        for (int e = 0; e < VEC; e++) xr[m][e] = own.e[e];
      }
      // the halo row, by the threads with the fewest vectors of their own
      if (co.c1 != 0.f) {
        const int ih = halo_row(co.c1);
        T* const hrow = co.c1 > 0.f ? stage : sb + rows * pitch;
        for (int v = NT - 1 - tid; v < QV; v += NT) {
          Vec<T> o;
#pragma unroll
          for (int e = 0; e < VEC; e++) o.e[e] = (T)0;
          if (ih >= 0) {
            const T axh = co.c1 > 0.f ? ax_above : ax_below;
            const int ku = ih < gm.i_neg ? k + 1 : k - 1;
            Vec<T> u = o;
            if (ku >= 0 && ku < nx)
              u = *reinterpret_cast<const Vec<T>*>(sb + (rows + 1) * pitch + v * VEC);
            else if (ku < 0)
              u = wall_inflow(ih, v * VEC);
            o = *reinterpret_cast<const Vec<T>*>(hrow + v * VEC);
#pragma unroll
            for (int e = 0; e < VEC; e++) o.e[e] = x_step(o.e[e], u.e[e], axh, (T)1 - axh);
          }
          *reinterpret_cast<Vec<T>*>(hrow + v * VEC) = o;
        }
      }
    }
    fence_proxy_async_smem();  // the stage's next contents come by a bulk copy
    ok = __syncthreads_and(ok);
    if (!ok) break;
    // every thread is past plane q - 1: its stage and its warp sums are whole
    if (tid == 0 && q > 0 && q - 1 + NS < n_items) {
      issue(q - 1 + NS, c1_issue);
      if (q + NS < n_items) c1_issue = a.c1_32[plane_of(q + NS)];
    }
    if (q > 0 && s_first + q - 1 >= s0 && warp == q % NW) fold(plane_of(q - 1), (q - 1) & 1);
    if (prime) continue;

    // ---- velocity step of g, x-step of the result
    const bool band = k >= band_lo && k < band_hi;
    const bool store = s_first + q >= s0;
    // a Strang step's x = 0 plane of rows with v1 > 0 waits for its inflow
    const bool deferred = STRANG && k == 0 && dir > 0;
    const bool edge = STRANG && ((k == 0 && dir < 0) || (k == nx - 1 && dir > 0));
    const int nboff = co.c1 > 0.f ? -pitch : (co.c1 < 0.f ? pitch : 0);
    const double dd = d2 - (double)(BGK ? co.ba + a1 : a1);  // FP64: 1 - |c_2| - |c_1| - dt nu
    if (store && warp == (q + 3) % NW) {
      const int erow = co.c1 > 0.f && i1 == nv1 ? rows - 1 : (co.c1 < 0.f && i0 == 0 ? 0 : -1);
      edge_loss(k, sb, erow, a1);
    }
    T sum_n = (T)0;
    F2 sum2 = f2_pack(0.f, 0.f);
    float sh_ = 0.f, sc_ = 0.f, sl_ = 0.f;  // FP64 grids: compensated FP32 sum
    T* const oplane = fout + (size_t)k * plane + (size_t)i0 * pitch + so0;
    // ANY: a plane with the source, at a boundary or only on the way to the
    // chunk's first one; else a plane with none of these
    auto velocity = [&](auto any) {
      constexpr bool ANY = decltype(any)::value;
#pragma unroll
      for (int m = 0; m < M; m++) {
        if (NT * m >= nvec) break;
        const bool in = flg >> m & 1;
        const int so = so0 + NT * VEC * m;
        const T* const c = sb + (in ? so : 0);
        const Vec<T> g = *reinterpret_cast<const Vec<T>*>(c);
        const Vec<T> nb = *reinterpret_cast<const Vec<T>*>(c + nboff);
        // v2 upwind (c_2 >= 0 since E_y <= 0): element j - 1
        T left;
        if constexpr (sizeof(T) == 4) {
          left = c[-1];
        } else {  // (a load of every lane took Lie steps of FP64 grids 11 % longer)
          left = __shfl_up_sync(0xffffffffu, g.e[VEC - 1], 1);
          if (lane == 0) left = c[-1];
        }
        if (flg >> (8 + m) & 1) left = (T)0;
        Vec<T> s, out;
#pragma unroll
        for (int e = 0; e < VEC; e++) s.e[e] = (T)0;
        if (ANY && band && in) {
          const int r = row_of(m);
          if constexpr (sizeof(T) == 4) {
            const T sr = srow[r];
            const Vec<T> sc = *reinterpret_cast<const Vec<T>*>(scol + (so - r * pitch));
#pragma unroll
            for (int e = 0; e < VEC; e++) s.e[e] = sr * sc.e[e];
          } else {
            s = *reinterpret_cast<const Vec<T>*>(a.tab.src + (size_t)i0 * pitch + so);
          }
        }
        if (BGK && in) {  // gain dt nu_k n_k m1[i] m2[j] of the collision term
          const int r = row_of(m);
          const T ms = co.bs * m1[r];
          const Vec<T> mv = *reinterpret_cast<const Vec<T>*>(m2 + (so - r * pitch));
#pragma unroll
          for (int e = 0; e < VEC; e++) s.e[e] = fma(ms, mv.e[e], s.e[e]);
        }
        if constexpr (sizeof(T) == 4) {  // two cells to an instruction
          const F2 a1p = f2_pack(a1, a1), a2p = f2_pack(a2, a2);
          const F2 g0 = f2_pack(g.e[0], g.e[1]), g1 = f2_pack(g.e[2], g.e[3]);
          F2 s0 = f2_pack(s.e[0], s.e[1]), s1 = f2_pack(s.e[2], s.e[3]);
          if (BGK) {
            const F2 ba = f2_pack(-co.ba, -co.ba);
            s0 = f2_fma(ba, g0, s0);
            s1 = f2_fma(ba, g1, s1);
          }
          s0 = f2_fma(a1p, f2_sub(f2_pack(nb.e[0], nb.e[1]), g0), s0);
          s1 = f2_fma(a1p, f2_sub(f2_pack(nb.e[2], nb.e[3]), g1), s1);
          s0 = f2_fma(a2p, f2_pack(left - g.e[0], g.e[0] - g.e[1]), s0);
          s1 = f2_fma(a2p, f2_pack(g.e[1] - g.e[2], g.e[2] - g.e[3]), s1);
          const float2 h0 = f2_unpack(f2_add(g0, s0)), h1 = f2_unpack(f2_add(g1, s1));
          out.e[0] = h0.x;
          out.e[1] = h0.y;
          out.e[2] = h1.x;
          out.e[3] = h1.y;
        } else {
#pragma unroll
          for (int e = 0; e < VEC; e++) {
            const T w = e == 0 ? left : g.e[e == 0 ? 0 : e - 1];
            out.e[e] = fma(a2, w, fma(a1, nb.e[e], fma(dd, g.e[e], s.e[e])));
          }
        }
        if (padded && (flg >> (16 + m) & 1)) {  // row padding stays zero
#pragma unroll
          for (int e = 1; e < VEC; e++)
            if (e > last_e) out.e[e] = (T)0;
        }
        if constexpr (STRANG) {
          if (ANY && edge && in) *reinterpret_cast<Vec<T>*>(static_cast<T*>(sa.h_wall) + (size_t)i0 * pitch + so) = out;
          const Vec<T> h = out;
          if (!ANY || !deferred)
            out = x_step_vec(h, hr[m], ax[m], sizeof(T) == 8 ? srow[row_of(m)] : (T)0);
#pragma unroll
          for (int e = 0; e < VEC; e++) hr[m][e] = h.e[e];
        }
        if ((ANY && !store) || !in) continue;
        if constexpr (sizeof(T) == 4) {
          sum2 = f2_add(sum2, f2_add(f2_pack(out.e[0], out.e[1]), f2_pack(out.e[2], out.e[3])));
        } else {
#pragma unroll
          for (int e = 0; e < VEC; e++) {
            float hi, lo;
            split_double((double)out.e[e], hi, lo);
            two_sum_acc(sh_, sc_, hi);
            sl_ += lo;
          }
        }
        if (in_bounds(k >= 0 && k < nx, a.st))
          __stcs(reinterpret_cast<float4*>(oplane + NT * VEC * m), *reinterpret_cast<const float4*>(&out));
      }
    };
    if (band || !store || deferred || edge)
      velocity(std::true_type());
    else
      velocity(std::false_type());
    if constexpr (sizeof(T) == 4) {
      const float2 s2 = f2_unpack(sum2);
      sum_n = s2.x + s2.y;
    }
    // the plane's warp sums
    if constexpr (sizeof(T) == 4) {
      const T ws = warp_sum(sum_n);
      if (lane == 0) sh.wn[q & 1][warp] = make_float2(ws, 0.f);
    } else {
      float lo = sc_ + sl_;
      for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_down_sync(0xffffffffu, sh_, o);
        const float ol = __shfl_down_sync(0xffffffffu, lo, o);
        float c = 0.f;
        two_sum_acc(sh_, c, oh);
        lo += ol + c;
      }
      if (lane == 0) sh.wn[q & 1][warp] = make_float2(sh_, lo);
    }
  }
  if (!ok) {  // a wait ran out: the copies in flight land before the CTA leaves
    if (tid == 0) {
      atomicOr(&a.st->flags, kFlagTimeout);
      for (int u = q; u < min(n_items, max(q - 1, 0) + NS); u++)
        if (u != withheld) mbar_wait(&sh.full[u % NS], (uint32_t)((u / NS) & 1), wlim);
    }
    return;
  }
  // ---- the last plane's sums; the boundary plane's flux sums
  const bool tail = s1 == nx;
  if (tail) {
    double b3[3];
    bool neg = false;
    if (STRANG) {
      neg = wall_terms_ahead<T, false>(static_cast<const T*>(sa.h_wall), a.tab, tid, NT, i0, rows,
                                       pitch, dir < 0, b3);
      if (lane == 0)
        for (int i = 0; i < 3; i++) sh.wall[0][warp][i] = b3[i];
    }
    const int k = plane_of(n_items - 1);
    neg |= wall_terms_ahead<T, false>(fout + (size_t)k * plane, a.tab, tid, NT, i0, rows, pitch,
                                      dir < 0, b3);
    if (lane == 0)
      for (int i = 0; i < 3; i++) sh.wall[1][warp][i] = b3[i];
    if (__any_sync(0xffffffffu, neg) && lane == 0) atomicOr(&a.st->flags, kFlagNegative);
  }
  __syncthreads();
  if (warp == 0) fold(plane_of(n_items - 1), (n_items - 1) & 1);
  if (tail && warp == 1 && lane < 6) {
    const int b = lane / 3, i = lane % 3;
    if (b == 1 || STRANG) {
      double s = 0.0;
      for (int w = 0; w < NW; w++) s += sh.wall[b][w][i];
      double* const dst = b ? (i == 0 ? a.part.pe : (i == 1 ? a.part.see : a.part.vac))
                            : (i == 0 ? sa.pe_mid : (i == 1 ? sa.see_mid : sa.vac_mid));
      dst[t] = s;
    }
  }
}

// Strang step, after the march: fold the boundary sums of the state h after
// the velocity step, add dt/2 of the fluxes to the ledger and the surface
// charge (Eqs. 12-14, 18; block 0), and complete the x = 0 plane of the rows
// with v1 > 0, which holds h, by the x-step over dt/2 with the inflow of those
// fluxes.  One block per tile of such rows: each folds the sums by itself, in
// the same order.
// A thread has one vector, loaded before the fold.
constexpr int kWallThreads = kSplitThreads * kSplitVec;
template <typename T>
__global__ void __launch_bounds__(kWallThreads) strang_wall_kernel(const __grid_constant__ SplitArgs sa) {
  constexpr int VEC = Vec<T>::N;
  __shared__ double s_see;
  __shared__ double wn[kWallThreads / 32];
  const StepArgs& a = sa.a;
  const Params& p = *a.prm;
  DevState* st = a.st;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, pitch = a.pitch;
  const int t = a.geom.t_neg + blockIdx.x;
  const double refl = p.refl;
  const int QV = pitch / VEC;
  T* const f = static_cast<T*>(a.f_out);  // the x = 0 plane
  bool in = false;
  Vec<T> o, mir;
  double gse[VEC];
  T cx = (T)0;
  size_t at = 0;
#pragma unroll
  for (int e = 0; e < VEC; e++) {
    o.e[e] = mir.e[e] = (T)0;
    gse[e] = 0.0;
  }
  if (t < a.geom.n_tiles) {
    int i0, i1, dir;
    tile_rows(a.geom, a.nv1, t, &i0, &i1, &dir);
    const int r = tid / QV, c = (tid - r * QV) * VEC, i = i0 + r;
    in = i < i1;
    if (in) {
      at = (size_t)i * pitch + c;
      cx = sizeof(T) == 8 ? (T)a.tab.cx[i] : (T)a.tab.cx32[i];
      o = *reinterpret_cast<const Vec<T>*>(f + at);
#pragma unroll
      for (int e = 0; e < VEC; e += 2) {
        const double2 g = *reinterpret_cast<const double2*>(a.tab.gse + at + e);
        gse[e] = g.x;
        gse[e + 1] = g.y;
      }
      if (refl > 0.0)
        mir = *reinterpret_cast<const Vec<T>*>(static_cast<const T*>(sa.h_wall) +
                                               (size_t)(a.nv1 - 1 - i) * pitch + c);
    }
  }
  if (warp == 0) {
    double pe = 0.0, see = 0.0, vac = 0.0;
    for (int u = lane; u < a.part.nu; u += 32) {
      pe += sa.pe_mid[u];
      see += sa.see_mid[u];
      vac += sa.vac_mid[u];
    }
    pe = warp_sum(pe);
    see = warp_sum(see);
    vac = warp_sum(vac);
    if (lane == 0) {
      pe *= p.dvv;
      see = p.see_enabled ? see * p.dvv * (1.0 - p.refl) : 0.0;
      vac *= p.dvv;
      s_see = see;
      if (blockIdx.x == 0 && st->flags == 0) {
        const double h = 0.5 * p.dt;
        st->cum_emit += h * (see + p.refl * pe);
        st->cum_see += h * see;
        st->cum_pe += h * pe;
        st->cum_vac += h * vac;
        st->sigma += kQe * h * (see - (1.0 - p.refl) * pe);
      }
    }
  }
  // a sticky error freezes the state
  if (__syncthreads_or(tid == 32 && *const_cast<volatile unsigned*>(&st->flags) != 0)) return;
  T sum = (T)0, err = (T)0;
  if (in) {
    const double gsee = s_see;
#pragma unroll
    for (int e = 0; e < VEC; e++) {
      double g = gsee * gse[e];
      if (refl > 0.0) g = fma(refl, (double)mir.e[e], g);
      o.e[e] = x_step(o.e[e], (T)g, (T)0.5 * cx, (T)1 - (T)0.5 * cx);
      const T s = sum + o.e[e], b = s - sum;  // TwoSum
      err += (sum - (s - b)) + (o.e[e] - b);
      sum = s;
    }
    *reinterpret_cast<Vec<T>*>(f + at) = o;
  }
  double n = sizeof(T) == 8 ? (double)(sum + err) : (double)sum + (double)err;
  n = warp_sum(n);
  if (lane == 0) wn[warp] = n;
  __syncthreads();
  if (warp == 0 && t < a.geom.n_tiles) {
    n = warp_sum(wn[lane]);
    if (lane == 0) a.part.n[t] = n;  // plane 0
  }
}

template <typename T, bool STRANG, bool BGK>
cudaError_t fit_split(int optin, size_t smem, int* best) {
  int n = 0;
  cudaError_t e = cudaFuncSetAttribute(split_kernel<T, STRANG, BGK>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, split_kernel<T, STRANG, BGK>, kSplitThreads, smem);
  if (e == cudaSuccess) *best = std::min(*best, n);
  return e;
}
// CTAs on an SM, the fewer of the variants with and without collisions
template <typename T>
int split_ctas_per_sm(size_t smem, bool strang) {
  int dev = 0, optin = 0, best = 1 << 30;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      smem > (size_t)optin)
    return 0;
  const cudaError_t e0 = strang ? fit_split<T, true, false>(optin, smem, &best)
                                : fit_split<T, false, false>(optin, smem, &best);
  const cudaError_t e1 = strang ? fit_split<T, true, true>(optin, smem, &best)
                                : fit_split<T, false, true>(optin, smem, &best);
  if (e0 != cudaSuccess || e1 != cudaSuccess)
    return 0;
  return best;
}

template <typename T>
cudaError_t launch_typed(const SplitArgs& sa, bool strang, bool bgk, cudaStream_t s) {
  const Geom& gm = sa.a.geom;
  const int grid = gm.n_tiles * gm.n_chunks;
  const size_t smem = split_smem_bytes<T>(gm.stage_elems, sa.a.pitch);
  if (!strang) {
    if (bgk)
      split_kernel<T, false, true><<<grid, kSplitThreads, smem, s>>>(sa);
    else
      split_kernel<T, false, false><<<grid, kSplitThreads, smem, s>>>(sa);
    return cudaGetLastError();
  }
  if (bgk)
    split_kernel<T, true, true><<<grid, kSplitThreads, smem, s>>>(sa);
  else
    split_kernel<T, true, false><<<grid, kSplitThreads, smem, s>>>(sa);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  strang_wall_kernel<T><<<std::max(1, gm.n_tiles - gm.t_neg), kWallThreads, 0, s>>>(sa);
  return cudaGetLastError();
}

// Whether one march is faster than the passes.  Its planes are a chain of two
// phases each, which the passes' pipeline of planes has not, so it loses where
// a chunk has many planes and a plane little work or twice the reads:
//  - tiles of two rows, whose halo rows double the reads (us a step, march and
//    passes: Lie FP32 64 x 64 x 2000, 17 planes a chunk, 54 and 56; 256 x 64 x
//    2000, 65 planes, 157 and 119; FP64 64 x 64 x 1000, 17 planes, 130 and 115,
//    16 x 32 x 1000, 2 planes, 32 and 58; Strang FP64 64 x 64 x 1000 166 and
//    168, 256 x 64 x 1000, 65 planes, 536 and 477; Strang FP32 256 x 64 x 2000
//    169 and 187);
//  - thin grids, whose passes run as half units (Lie FP32 1024 x 16 x 16, 5
//    planes, 24.3 and 26.9; 2048 x 16 x 16, 9 planes, 32.9 and 31.5; 8192 x 16 x
//    16, 36 planes, 87 and 72; FP64, bound by its pipe sooner: 2048 x 32 x 32, a
//    vector a thread, 61 and 69; 2048 x 8 x 8 60 and 45).
bool march_pays(bool f32, bool strang, bool half, int most_rows, int vectors, int planes) {
  if (most_rows == 2) return strang ? f32 || planes <= 16 : planes <= (f32 ? 17 : 6);
  if (!half) return true;
  if (f32) return planes <= (vectors < 128 ? 8 : strang ? 14 : 9);
  if (vectors >= (strang ? 128 : 256)) return true;
  return planes <= (strang || vectors >= 64 ? 8 : 4);
}

}  // namespace

bool plan_split(int precision, bool strang, int nx, int nv1, int pitch, int i_neg, bool half,
                int sms, Geom* gm) {
  const int vec = precision == FK_F32 ? 4 : 2;
  const int most = std::min(kSplitThreads * kSplitVec * vec / pitch, kMaxTileRows);
  if (most < 2) return false;  // the halo rows would double the reads
  Geom m{};
  m.i_neg = i_neg;
  auto split = [&](int rows, int* nt, int* ti) {
    *nt = (rows + most - 1) / most;
    *ti = *nt ? (rows + *nt - 1) / *nt : 1;
  };
  int t_pos = 0;
  split(i_neg, &m.t_neg, &m.ti_neg);
  split(nv1 - i_neg, &t_pos, &m.ti_pos);
  m.n_tiles = m.t_neg + t_pos;
  // a tile, its v1 halo rows above and below, and a halo row's x neighbour
  m.stage_elems = (std::max(m.ti_neg, m.ti_pos) + 3) * pitch;
  const int per_sm = precision == FK_F32
                         ? split_ctas_per_sm<float>(split_smem_bytes<float>(m.stage_elems, pitch), strang)
                         : split_ctas_per_sm<double>(split_smem_bytes<double>(m.stage_elems, pitch), strang);
  if (per_sm < 1) return false;
  // one wave of units; the last chunk is shorter by what its boundary sums cost
  const int nc = std::max(1, std::min(sms * per_sm / m.n_tiles, nx / kSplitMinChunk));
  const int last = std::min(kSplitLast, (nx + nc - 1) / nc - 1);
  m.chunk_len = (nx + last + nc - 1) / nc;
  m.n_chunks = (nx + m.chunk_len - 1) / m.chunk_len;
  *gm = m;
  return march_pays(precision == FK_F32, strang, half, most,
                    std::max(m.ti_neg, m.ti_pos) * (pitch / vec), m.chunk_len);
}

cudaError_t launch_split_step(const SplitArgs& sa, int precision, bool strang, bool bgk,
                              cudaStream_t s) {
  return precision == FK_F32 ? launch_typed<float>(sa, strang, bgk, s)
                             : launch_typed<double>(sa, strang, bgk, s);
}

}  // namespace fk
