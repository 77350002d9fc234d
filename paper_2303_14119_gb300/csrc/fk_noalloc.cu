// fk_density_moment_noalloc: the density moment n_e(x) of a distribution
// that already lives in device memory, computed without allocating any
// memory.  Its scratch (the per-plane partial sums of a two-pass,
// fixed-order reduction) is a file-scope __device__ array of fixed size
// that every GPU loading this library holds until the process exits.
#include <stdint.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "fk_internal.cuh"
#include "fk_sum.cuh"

namespace {

constexpr int kUnits = 16;  // most partial sums per x-plane
constexpr int kTwoBlocksPerSm = 2 * 152;  // on GB300

// Scratch shared by every call: FK_NOALLOC_MAX_PARTIALS doubles (1 MiB).
static __device__ __align__(256) double g_noalloc_partials[FK_NOALLOC_MAX_PARTIALS];

// In host code the name g_noalloc_partials is only a host-side stand-in;
// the kernels get the device address looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_mutex;
double* g_scratch[kMaxDevices] = {};

// Pass 1: block (k, u) sums its slice of plane k, kGroup values of a thread at
// a time (fk_sum.cuh), in a fixed order.  16-byte loads, eight in flight a
// thread; a slice that starts off a 16-byte boundary takes its first value
// apart.  With one slice a plane the sum is the result (n_e).
//
// Bound by HBM: 1024 planes of 256 x 256 take 83 us (6.4 TB/s); with an FP64
// addition for each 8-byte load they took 179 + 5 us.
template <int kThreads>
__global__ void __launch_bounds__(kThreads)
moment_partials(const double* __restrict__ f, long long plane, int units, double* partials,
                double dvv, double* n_e) {
  __shared__ double sh[kThreads / 32];
  const int k = blockIdx.x / units, u = blockIdx.x - (blockIdx.x / units) * units;
  const long long per = (plane + units - 1) / units;
  const long long lo = (long long)u * per;
  const long long hi = lo + per < plane ? lo + per : plane;
  const double* p = f + (long long)k * plane + lo;
  long long n = hi > lo ? hi - lo : 0;
  double s = 0.0;
  if (n > 0 && ((uintptr_t)p & 15)) {
    if (threadIdx.x == 0) s = p[0];
    p += 1;
    n -= 1;
  }
  const double2* p2 = reinterpret_cast<const double2*>(p);
  const long long n2 = n / 2;
  for (long long c0 = threadIdx.x; c0 - threadIdx.x < n2; c0 += kThreads * (fk::kGroup / 2)) {
    double x[fk::kGroup];
#pragma unroll
    for (int j = 0; j < fk::kGroup / 2; j++) {
      const long long c = c0 + (long long)j * kThreads;
      const double2 v = c < n2 ? __ldcs(p2 + c) : make_double2(0.0, 0.0);
      x[2 * j] = v.x;
      x[2 * j + 1] = v.y;
    }
    s = fk::add_group(x, s);
  }
  if ((n & 1) && threadIdx.x == 0) s += p[n - 1];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kThreads / 32; w++) t += sh[w];
    if (units == 1)
      n_e[k] = t * dvv;
    else
      partials[blockIdx.x] = t;  // every slot used by this call is written here
  }
}

// Pass 2: n_e[k] = dv1 dv2 * (sum of plane k's partials, in unit order).
__global__ void moment_finish(const double* partials, int nx, int units, double dvv,
                              double* n_e) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nx) return;
  double s = 0.0;
  for (int u = 0; u < units; u++) s += partials[k * units + u];
  n_e[k] = s * dvv;
}

}  // namespace

extern "C" fk_status fk_density_moment_noalloc(const double* f_dev, int32_t nx, int32_t nv1,
                                               int32_t nv2, double dv1, double dv2,
                                               double* n_e_dev, void* cuda_stream) {
  if (!f_dev || !n_e_dev) {
    fk::set_thread_error("fk_density_moment_noalloc: f and n_e must be device pointers");
    return FK_EINVAL;
  }
  if (nx < 1 || nv1 < 1 || nv2 < 1 || !(dv1 > 0.0) || !(dv2 > 0.0)) {
    fk::set_thread_error("fk_density_moment_noalloc: need nx, nv1, nv2 >= 1 and dv1, dv2 > 0");
    return FK_EINVAL;
  }
  if ((long long)nx * kUnits > FK_NOALLOC_MAX_PARTIALS) {
    fk::set_thread_error(("fk_density_moment_noalloc: nx = " + std::to_string(nx) +
                          " exceeds the scratch limit of " +
                          std::to_string(FK_NOALLOC_MAX_PARTIALS / kUnits) + " planes")
                             .c_str());
    return FK_EINVAL;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    fk::set_thread_error("fk_density_moment_noalloc: no usable current CUDA device");
    return FK_ECUDA;
  }
  double* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mutex);
    if (!g_scratch[dev]) {
      // first call on this device (with it current): look up the device
      // address of the scratch array
      void* ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_noalloc_partials);
      if (e != cudaSuccess) {
        fk::set_thread_error((std::string("fk_density_moment_noalloc: cudaGetSymbolAddress: ") +
                              cudaGetErrorString(e))
                                 .c_str());
        return FK_ECUDA;
      }
      g_scratch[dev] = static_cast<double*>(ptr);
    }
    scratch = g_scratch[dev];
  }
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const long long plane = (long long)nv1 * nv2;
  // One block a plane where the second launch (4 us) costs more than the idle SMs:
  // from 64 planes on (64 of 200 x 200 take 10 us either way, 32 of 256 x 256
  // 16.5 us whole and 12.3 in slices), and for small planes (16 of 64 x 64: 4.5
  // against 10.4 us; 2 of 256 x 256: 12.6 against 8.8).  Large planes that leave
  // SMs idle are worth the launch (64 of 512 x 512: 48 whole, 29 in four slices;
  // 64 of 1024 x 1024: 166 and 87; 300 of 512 x 512: the same).  512 threads
  // where they have more than two groups of values each (1024 planes of 256 x
  // 256: 83 against 92 us), else 256 (669 planes of 112 x 129: 16 against 18 us).
  int units = std::min(kUnits, (kTwoBlocksPerSm + nx - 1) / nx);
  if (plane <= 128 * 128)
    units = 1;
  else if (nx >= 64)
    units = plane >= 512 * 512 && nx < kTwoBlocksPerSm ? 4 : 1;
  const double dvv = dv1 * dv2;
  if (plane / units >= 2 * 512 * fk::kGroup)
    moment_partials<512><<<nx * units, 512, 0, s>>>(f_dev, plane, units, scratch, dvv, n_e_dev);
  else
    moment_partials<256><<<nx * units, 256, 0, s>>>(f_dev, plane, units, scratch, dvv, n_e_dev);
  if (units > 1)
    moment_finish<<<(nx + 255) / 256, 256, 0, s>>>(scratch, nx, units, dvv, n_e_dev);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    fk::set_thread_error((std::string("fk_density_moment_noalloc: launch: ") +
                          cudaGetErrorString(e))
                             .c_str());
    return FK_ECUDA;
  }
  return FK_OK;
}
