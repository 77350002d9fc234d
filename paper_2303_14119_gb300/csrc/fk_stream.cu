// Kernels and launchers of the streaming step: one grid, or many grids in one
// launch, with whole-CTA or half-CTA units (fk_stream_unit.cuh holds the unit).
#include "fk_stream_unit.cuh"

namespace fk {

namespace {

// One grid, whole-CTA units: CTA b runs tile b % n_tiles of chunk
// b / n_tiles.
template <typename T, bool PADDED, bool BGK>
__global__ void __launch_bounds__(kBlock, 2) step_stream_kernel(const __grid_constant__ StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int nt = a.geom.n_tiles;
  stream_unit<T, PADDED, BGK, kThreads, false>(a, blockIdx.x % nt, blockIdx.x / nt, smem + kArgsBytes,
                                        threadIdx.x, 0);
}

// One grid, half units: CTA b runs units 2b and 2b + 1 on its two halves,
// each in a region of half_region_bytes.
template <typename T, bool PADDED, bool BGK>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? 3 : 2)
step_stream_half_kernel(const __grid_constant__ StepArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int nt = a.geom.n_tiles;
  const int h = threadIdx.x / kHalfBlock;
  const int u = 2 * blockIdx.x + h;
  if (u >= nt * a.geom.n_chunks) return;
  unsigned char* region = smem + h * half_region_bytes<T>(a.geom.stage_elems, a.pitch);
  stream_unit<T, PADDED, BGK, kHalfThreads, false>(a, u % nt, u / nt, region + kArgsBytes,
                                            threadIdx.x - h * kHalfBlock, 1 + h);
}

// Many grids in one launch, whole-CTA units: CTA b copies the arguments of
// grid units[b].x into the slot at the start of its shared memory and runs
// that grid's unit units[b].y = tile + n_tiles * chunk.
template <typename T, bool PADDED, bool BGK>
__global__ void __launch_bounds__(kBlock, 2)
step_stream_batch_kernel(const BatchInst* __restrict__ inst, const int2* __restrict__ units) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int2 u = units[blockIdx.x];
  const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&inst[u.x].a);
  unsigned long long* dst = reinterpret_cast<unsigned long long*>(smem);
  for (int w = threadIdx.x; w < (int)(sizeof(StepArgs) / 8); w += blockDim.x) dst[w] = src[w];
  __syncthreads();
  const StepArgs& a = *reinterpret_cast<const StepArgs*>(smem);
  const int nt = a.geom.n_tiles;
  stream_unit<T, PADDED, BGK, kThreads, true>(a, u.y % nt, u.y / nt, smem + kArgsBytes, threadIdx.x, 0);
}

// Many grids in one launch, half units: CTA b runs unit pairs[b].y of grid
// pairs[b].x on threads [0, kHalfBlock) and unit pairs[b].w of grid
// pairs[b].z (none if pairs[b].z < 0) on the rest, each half in a region of
// half_bytes whose slot receives that grid's arguments.
template <typename T, bool PADDED, bool BGK>
__global__ void __launch_bounds__(kBlock, sizeof(T) == 4 ? 3 : 2)
step_stream_batch_half_kernel(const BatchInst* __restrict__ inst, const int4* __restrict__ pairs,
                              int half_bytes) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int4 c = pairs[blockIdx.x];
  const int h = threadIdx.x / kHalfBlock, ht = threadIdx.x - h * kHalfBlock;
  const int g = h ? c.z : c.x, u = h ? c.w : c.y;
  unsigned char* region = smem + (size_t)h * half_bytes;
  if (g >= 0) {
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&inst[g].a);
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(region);
    for (int w = ht; w < (int)(sizeof(StepArgs) / 8); w += kHalfBlock) dst[w] = src[w];
  }
  __syncthreads();
  if (g < 0) return;  // the idle half of a CTA with one unit
  const StepArgs& a = *reinterpret_cast<const StepArgs*>(region);
  const int nt = a.geom.n_tiles;
  stream_unit<T, PADDED, BGK, kHalfThreads, true>(a, u % nt, u / nt, region + kArgsBytes, ht, 1 + h);
}

// FP32 grids with collisions take the kernel for padded rows, whose rows may
// also have no padding: the compiler keeps it within its registers, the other
// one spilled 32 bytes in its march (batches of unpadded grids, us a step: four
// of 1024 x 128 x 128 150 -> 132, three of 512 x 256 x 256 200 -> 179, twelve of
// a sweep 127 -> 112; before the two-cell update 147, 191 and 124).
template <typename T, bool PADDED, bool BGK>
constexpr auto batch_kernel() {
  return step_stream_batch_kernel<T, PADDED || (BGK && sizeof(T) == 4), BGK>;
}

}  // namespace

int stream_tile_rows(int precision, int pitch, int smem_per_sm, int reserved_per_block,
                     bool half) {
  const int esize = precision == FK_F32 ? 4 : 8;
  const int vec = 16 / esize;
  const int cells = half ? kHalfThreads * (esize == 4 ? unit_vectors<kHalfThreads, 4>()
                                                    : unit_vectors<kHalfThreads, 8>()) * vec
                         : kThreads * kVecPerThread * vec;
  if (pitch > cells) return 0;
  int rows = cells / pitch;
  if (rows > kMaxTileRows) rows = kMaxTileRows;
  // two CTAs per SM: each unit holds its stages (kStages, or kHalfStages for
  // a half unit) of (rows + 1) * pitch elements (a half unit gets half of
  // its CTA, less the region's rounding)
  const int ns = half ? kHalfStages : kStages;
  const long tail =
      (long)(precision == FK_F32
                 ? (half ? tail_bytes<float, kHalfStages>(pitch) : tail_bytes<float, kStages>(pitch))
                 : (half ? tail_bytes<double, kHalfStages>(pitch)
                         : tail_bytes<double, kStages>(pitch)));
  const long cta = (long)smem_per_sm / 2 - reserved_per_block;
  const long budget = (half ? cta / 2 - 127 : cta) - tail;
  const long stage = budget / ns / 128 * 128;
  const long fit = stage / ((long)pitch * esize) - 1;  // one halo slot per stage
  if (fit < rows) rows = (int)fit;
  return rows > 0 ? rows : 0;
}

size_t stream_smem_bytes(int precision, int stage_elems, int pitch) {
  return precision == FK_F32 ? unit_smem_bytes<float, kStages>(stage_elems, pitch)
                             : unit_smem_bytes<double, kStages>(stage_elems, pitch);
}

size_t stream_half_bytes(int precision, int stage_elems, int pitch) {
  return precision == FK_F32 ? half_region_bytes<float>(stage_elems, pitch)
                             : half_region_bytes<double>(stage_elems, pitch);
}

size_t stream_cta_smem_bytes(int precision, const Geom& gm, int pitch) {
  return gm.half ? 2 * stream_half_bytes(precision, gm.stage_elems, pitch)
                 : stream_smem_bytes(precision, gm.stage_elems, pitch);
}

namespace {
// allow the device's largest opt-in shared memory for kernel k and ask how
// many CTAs of smem_bytes fit on an SM
// allow the device's largest opt-in shared memory for kernel k and ask how
// many CTAs of smem_bytes fit on an SM; *best keeps the smallest answer of
// the kernels that count (count = false: the attribute is only set)
template <typename K>
cudaError_t fit_kernel(K k, int optin, size_t smem_bytes, bool count, int* best) {
  int n = 0;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kBlock, smem_bytes);
  if (e == cudaSuccess && count && n < *best) *best = n;
  return e;
}
template <typename T, bool P, bool B>
cudaError_t fit_four(int optin, size_t smem_bytes, bool whole, bool half, int* best) {
  cudaError_t e = fit_kernel(step_stream_kernel<T, P, B>, optin, smem_bytes, whole, best);
  if (e == cudaSuccess) e = fit_kernel(batch_kernel<T, P, B>(), optin, smem_bytes, whole, best);
  if (e == cudaSuccess) e = fit_kernel(step_stream_half_kernel<T, P, B>, optin, smem_bytes, half, best);
  if (e == cudaSuccess)
    e = fit_kernel(step_stream_batch_half_kernel<T, P, B>, optin, smem_bytes, half, best);
  return e;
}
template <typename T>
int ctas_per_sm(int optin, size_t smem_bytes, int layout) {
  const bool whole = layout != kLayoutHalf, half = layout != kLayoutWhole;
  int best = 1 << 30;
  cudaError_t e = fit_four<T, false, false>(optin, smem_bytes, whole, half, &best);
  if (e == cudaSuccess) e = fit_four<T, true, false>(optin, smem_bytes, whole, half, &best);
  if (e == cudaSuccess) e = fit_four<T, false, true>(optin, smem_bytes, whole, half, &best);
  if (e == cudaSuccess) e = fit_four<T, true, true>(optin, smem_bytes, whole, half, &best);
  return e == cudaSuccess ? best : 0;
}
}  // namespace

int stream_ctas_per_sm(int precision, size_t smem_bytes, int layout) {
  // the attribute is per kernel, shared by every grid and batch: allow the
  // device's largest opt-in size on every variant, and ask the occupancy of
  // this size (the smallest over the single-grid and batched variants of
  // the layout asked for; the half-unit kernels of FP32 grids fit more
  // CTAs on an SM than the whole-CTA ones)
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return 0;
  if (smem_bytes > (size_t)optin) return 0;
  return precision == FK_F32 ? ctas_per_sm<float>(optin, smem_bytes, layout)
                             : ctas_per_sm<double>(optin, smem_bytes, layout);
}

namespace {
template <typename T, bool BGK>
void launch_single(const StepArgs& a, int grid, size_t smem, bool padded, bool half,
                   cudaStream_t s) {
  if (half) {
    if (padded)
      step_stream_half_kernel<T, true, BGK><<<grid, kBlock, smem, s>>>(a);
    else
      step_stream_half_kernel<T, false, BGK><<<grid, kBlock, smem, s>>>(a);
  } else {
    if (padded)
      step_stream_kernel<T, true, BGK><<<grid, kBlock, smem, s>>>(a);
    else
      step_stream_kernel<T, false, BGK><<<grid, kBlock, smem, s>>>(a);
  }
}
template <typename T, bool BGK>
void launch_batch(const BatchInst* inst, const int2* units, int n_units, size_t smem,
                  const int4* pairs, int n_pairs, int half_bytes, bool padded, cudaStream_t s) {
  if (n_units > 0) {
    if (padded)
      batch_kernel<T, true, BGK>()<<<n_units, kBlock, smem, s>>>(inst, units);
    else
      batch_kernel<T, false, BGK>()<<<n_units, kBlock, smem, s>>>(inst, units);
  }
  if (n_pairs > 0) {
    const size_t hs = 2 * (size_t)half_bytes;
    if (padded)
      step_stream_batch_half_kernel<T, true, BGK><<<n_pairs, kBlock, hs, s>>>(inst, pairs, half_bytes);
    else
      step_stream_batch_half_kernel<T, false, BGK><<<n_pairs, kBlock, hs, s>>>(inst, pairs, half_bytes);
  }
}
}  // namespace

cudaError_t launch_step_stream(const StepArgs& a, int precision, bool bgk, cudaStream_t s) {
  const int units = a.geom.n_tiles * a.geom.n_chunks;
  const bool half = a.geom.half != 0;
  const int grid = half ? (units + 1) / 2 : units;
  const size_t smem = stream_cta_smem_bytes(precision, a.geom, a.pitch);
  const bool padded = a.pitch != a.nv2;
  if (precision == FK_F32) {
    if (bgk)
      launch_single<float, true>(a, grid, smem, padded, half, s);
    else
      launch_single<float, false>(a, grid, smem, padded, half, s);
  } else {
    if (bgk)
      launch_single<double, true>(a, grid, smem, padded, half, s);
    else
      launch_single<double, false>(a, grid, smem, padded, half, s);
  }
  return cudaGetLastError();
}

cudaError_t launch_step_stream_batch(const BatchInst* inst, const int2* units, int n_units,
                                     const int4* pairs, int n_pairs, int precision, bool padded,
                                     bool bgk, size_t smem_bytes, int half_bytes,
                                     cudaStream_t s) {
  if (n_units <= 0 && n_pairs <= 0) return cudaSuccess;
  if (precision == FK_F32) {
    if (bgk)
      launch_batch<float, true>(inst, units, n_units, smem_bytes, pairs, n_pairs, half_bytes,
                                padded, s);
    else
      launch_batch<float, false>(inst, units, n_units, smem_bytes, pairs, n_pairs, half_bytes,
                                 padded, s);
  } else {
    if (bgk)
      launch_batch<double, true>(inst, units, n_units, smem_bytes, pairs, n_pairs, half_bytes,
                                 padded, s);
    else
      launch_batch<double, false>(inst, units, n_units, smem_bytes, pairs, n_pairs, half_bytes,
                                  padded, s);
  }
  return cudaGetLastError();
}

}  // namespace fk
