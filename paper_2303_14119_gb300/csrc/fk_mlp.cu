// Dense layers of the surface-charge surrogate on the tensor cores:
// C = A * B^T with bf16 A [M][K] and B [N][K] (both K-major), FP32
// accumulation in tensor memory (tcgen05.mma, operands in shared memory),
// and the epilogues the surrogate's training needs (bias, GELU and its
// derivative, bf16 copies in both layouts).
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include <string>

#include "fk_internal.cuh"
#include "fk_mlp.h"
#include "fk_mlp_internal.cuh"
#include "fk_tc.cuh"

namespace fk {

namespace {

constexpr int kMTile = 128;   // rows per CTA (one MMA M)
// columns per CTA (one MMA N at most): 64, or 32 where 64 leaves most SMs idle
constexpr int kNTileWide = 64, kNTileThin = 32;
constexpr int kNMax = 256;    // the largest N the entry points accept
constexpr int kKChunk = 64;   // K per stage (4 MMAs of K = 16)
constexpr int kGemmStages = 4;     // stages of the ring: K chunks in flight
constexpr int kGemmThreads = 256;  // 8 warps: two per 32-lane slice of tensor memory
constexpr int kCoreBytes = 128;    // one 8 x 16-byte core matrix
// a tile: [rows/8 row groups][kKChunk/8 K groups] core matrices
constexpr int kLboBytes = kCoreBytes;                        // next core matrix along K
constexpr int kSboBytes = (kKChunk / 8) * kCoreBytes;        // next 8-row group
constexpr int kATileBytes = kMTile * kKChunk * 2;            // 16 KB
constexpr int gemm_stage_bytes(int nt) { return kATileBytes + nt * kKChunk * 2; }  // 20 or 24 KB
// dynamic shared memory per CTA: the ring (two CTAs fit on an SM, with 2 x
// 64 of its 512 tensor-memory columns)
constexpr int gemm_smem(int nt) { return kGemmStages * gemm_stage_bytes(nt); }

__device__ __forceinline__ uint16_t f32_to_bf16(float x) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}
// GELU with the exact (erf) form and its derivative
__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) +
         z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// 16-byte asynchronous copy global -> shared (cp.async); zeros when !full
// (no byte of src is read then; src stays a valid address)
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool full) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst)), "l"(src),
               "r"(full ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// wait until at most n of this thread's copy groups are still pending
__device__ __forceinline__ void cp_async_wait(int n) {
  switch (n) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
  }
}

// Queue the copy of rows [r0, r0 + rows) x K columns [k0, k0 + kKChunk) of a
// K-major bf16 matrix into the core-matrix layout; zeros outside
// [0, nrows) x [0, K).
__device__ __forceinline__ void stage_tile(unsigned char* dst, const uint16_t* src, long long ld,
                                           int r0, int rows, int nrows, int k0, int K) {
  const int vecs = rows * (kKChunk / 8);
  for (int v = threadIdx.x; v < vecs; v += kGemmThreads) {
    const int r = v / (kKChunk / 8), kc = v - (v / (kKChunk / 8)) * (kKChunk / 8);
    const int gr = r0 + r, gk = k0 + kc * 8;
    const bool in = gr < nrows && gk < K;
    cp_async16(dst + ((r >> 3) * (kKChunk / 8) + kc) * kCoreBytes + (r & 7) * 16,
               in ? src + (long long)gr * ld + gk : src, in);
  }
}

// Bias gradients: sums over the batch of the bf16 rows [r0, r0 + kSumRows) of g.A,
// each as 256 strided FP32 sums folded in trees of 32 and of 8, one warp a row.
// (With 128 rows a CTA, sixteen a warp one after the other, they outlasted the
// products beside them: the gradient over 65536 rows of the 256-wide network took
// 8.4 ms, now 5.8; an epoch of 16384 in batches of 1024 3.1 and 2.5.)
constexpr int kSumRows = kGemmThreads / 32;
__device__ void row_sums_tile(const GemmArgs& g, int r0) {
  const int r = r0 + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r < g.M) {
    const uint16_t* row = g.A + (long long)r * g.lda;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int c0 = 0; c0 < g.sum_n; c0 += 256)
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const int c = c0 + 32 * j + lane;
        if (c < g.sum_n) acc[j] += __uint_as_float((uint32_t)row[c] << 16);
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int j = 0; j < 8; j++) acc[j] += __shfl_down_sync(0xffffffffu, acc[j], o);
    if (lane == 0)
      g.row_sum[r] = ((acc[0] + acc[4]) + (acc[2] + acc[6])) + ((acc[1] + acc[5]) + (acc[3] + acc[7]));
  }
}

// One CTA: rows [m0, m0 + 128) x columns [n0, n0 + Nc) of C.  The K chunks
// stream through a ring of kGemmStages shared-memory stages: every thread
// queues its part of a chunk's copies (cp.async) up to kGemmStages chunks
// ahead; once a chunk has landed, one thread issues its four MMAs and
// commits them to the stage's mbarrier, whose phase frees the stage for
// the chunk kGemmStages later.  Each output element sums its K terms in
// the same order whatever the grid, so results are deterministic.
//
// At the network's sizes (256 x 256 x 256) the MMAs are a few percent: what
// counts are the copies' latency and the epilogue, so eight warps share it,
// with 16-byte stores; the GELU layers took 26 us with four warps of 64 columns
// and one store an element.
//
// A launch holds up to three jobs (independent products, and the row sums of
// an operand), one after the other in the grid.
template <int kNTile>
__global__ void __launch_bounds__(kGemmThreads) gemm_tn_kernel(const __grid_constant__ GemmJobs jobs) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ uint64_t bar[kGemmStages];
  __shared__ uint32_t s_taddr;
  constexpr int kStageBytes = gemm_stage_bytes(kNTile);
  int cta = blockIdx.x, job = 0;
  while (cta >= jobs.ctas[job]) cta -= jobs.ctas[job++];
  const GemmArgs& g = jobs.g[job];
  if (g.row_sum) {  // uniform over the CTA
    row_sums_tile(g, cta * kSumRows);
    return;
  }
  const int mt = (g.M + kMTile - 1) / kMTile;
  const int m0 = (cta % mt) * kMTile;
  const int n0 = (cta / mt) * kNTile;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int N = g.N;
  const int Nc = min(kNTile, (N + 15) / 16 * 16 - n0);  // this CTA's columns, a multiple of 16
  const uint32_t ncols = Nc <= 32 ? 32u : 64u;
  if (warp == 0) {
    tc::tmem_alloc(&s_taddr, ncols);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int q = 0; q < kGemmStages; q++) tc::mbar_init(&bar[q], 1);
    tc::fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = s_taddr;
  const uint32_t idesc = tc::idesc_bf16_f32(kMTile, Nc);
  const int nch = (g.K + kKChunk - 1) / kKChunk;
  auto stage = [&](int c) {
    unsigned char* sA = smem + (c % kGemmStages) * kStageBytes;
    stage_tile(sA, g.A, g.lda, m0, kMTile, g.M, c * kKChunk, g.K);
    stage_tile(sA + kATileBytes, g.B, g.ldb, n0, Nc, N, c * kKChunk, g.K);
    cp_async_commit();
  };
  for (int c = 0; c < min(kGemmStages, nch); c++) stage(c);
  uint32_t parity = 0;  // bit q: the phase of stage q's mbarrier to wait for
  bool ok = true;
  for (int c = 0; c < nch && ok; c++) {
    const int q = c % kGemmStages;
    // chunk c's copies (later chunks' groups may still be in flight)
    cp_async_wait(min(nch, c + kGemmStages) - 1 - c);
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid == 0) {
      const uint32_t a0 = tc::smem_u32(smem + q * kStageBytes), b0 = a0 + kATileBytes;
      for (int kk = 0; kk < kKChunk / 16; kk++) {
        // K step of 16 = two core matrices along K
        const uint64_t ad = tc::smem_desc(a0 + kk * 2 * kLboBytes, kLboBytes, kSboBytes);
        const uint64_t bd = tc::smem_desc(b0 + kk * 2 * kLboBytes, kLboBytes, kSboBytes);
        tc::mma_bf16(taddr, ad, bd, idesc, (c > 0 || kk > 0) ? 1u : 0u);
      }
      tc::mma_commit(&bar[q]);
    }
    if (c + kGemmStages < nch || c == nch - 1) {
      // the stage is free (or, after the last chunk, D is complete) once
      // its MMAs have run
      ok = tc::mbar_wait(&bar[q], (parity >> q) & 1u);
      parity ^= 1u << q;
      tc::fence_after_sync();
      if (!__syncthreads_and(ok)) ok = false;
      if (ok && c + kGemmStages < nch) stage(c + kGemmStages);
    }
  }
  cp_async_wait(0);  // nothing left in flight into shared memory
  if (ok) {
    // epilogue: warps w and w + 4 hold rows m0 + 32 (w % 4) + lane (tensor-memory
    // lanes), 16 columns of every 32 each
    const int row = m0 + (warp & 3) * 32 + lane;
    const bool live = row < g.M;
    const bool whole = g.vec;  // 16-byte rows of C, H and Zin
    for (int c0 = (warp >> 2) * 16; c0 < Nc; c0 += 32) {
      uint32_t r[16];
      tc::tmem_ld16(taddr + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, r);
      tc::tmem_wait_ld();
      if (!live) continue;
      const int col0 = n0 + c0;
      float v[16];
#pragma unroll
      for (int e = 0; e < 16; e++) {
        v[e] = __uint_as_float(r[e]);
        if (g.epi != kEpiGeluBack && g.bias && col0 + e < N) v[e] += g.bias[col0 + e];
      }
      const bool full = whole && col0 + 16 <= N;
      if (g.epi != kEpiGeluBack) {
        float* crow = g.C + (long long)row * g.ldc + col0;
        if (full) {
#pragma unroll
          for (int e = 0; e < 16; e += 4)
            *reinterpret_cast<float4*>(crow + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        } else {
          for (int e = 0; e < 16 && col0 + e < N; e++) crow[e] = v[e];
        }
        if (g.epi == kEpiF32) continue;
      }
      float z[16];
      if (g.epi == kEpiGeluBack) {
        const float* zrow = g.Zin + (long long)row * g.ldz + col0;
        if (full) {
#pragma unroll
          for (int e = 0; e < 16; e += 4)
            *reinterpret_cast<float4*>(z + e) = *reinterpret_cast<const float4*>(zrow + e);
        } else {
#pragma unroll
          for (int e = 0; e < 16; e++) z[e] = col0 + e < N ? zrow[e] : 0.f;
        }
      }
      uint32_t h[8];  // bf16 pairs
#pragma unroll
      for (int e = 0; e < 16; e++) {
        float x = 0.f;
        if (row < g.m_valid) x = g.epi == kEpiBiasGelu ? gelu(v[e]) : v[e] * gelu_grad(z[e]);
        const uint32_t b = f32_to_bf16(x);
        if (e & 1)
          h[e / 2] |= b << 16;
        else
          h[e / 2] = b;
      }
      uint16_t* hrow = g.H + (long long)row * g.ldh + col0;
      if (full) {
        *reinterpret_cast<uint4*>(hrow) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4*>(hrow + 8) = make_uint4(h[4], h[5], h[6], h[7]);
      }
#pragma unroll
      for (int e = 0; e < 16; e++) {
        if (col0 + e >= N) break;
        const uint16_t x = (uint16_t)(h[e / 2] >> (16 * (e & 1)));
        if (!full) hrow[e] = x;
        if (g.Ht) g.Ht[(long long)(col0 + e) * g.ldht + row] = x;
      }
    }
  } else if (tid == 0) {
    atomicOr(g.err, 1);
    // a second bounded wait for MMAs still in flight before the memory is
    // freed: the last chunk's commit completes after every earlier one
    const int q = (nch - 1) % kGemmStages;
    tc::mbar_wait(&bar[q], (parity >> q) & 1u);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(taddr, ncols);
  }
}

// CTAs of a job with kNTile-column tiles
int job_ctas(const GemmArgs& g, int nt) {
  if (g.row_sum) return (g.M + kSumRows - 1) / kSumRows;
  return (g.M + kMTile - 1) / kMTile * (((g.N + 15) / 16 * 16 + nt - 1) / nt);
}

template <int kNTile>
cudaError_t launch_jobs(GemmJobs& jobs, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(gemm_tn_kernel<kNTile>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, gemm_smem(kNTile));
  if (e != cudaSuccess) return e;
  int total = 0;
  for (int j = 0; j < kGemmJobs; j++) {
    jobs.ctas[j] = j < jobs.n ? job_ctas(jobs.g[j], kNTile) : 0;
    total += jobs.ctas[j];
  }
  jobs.ctas[jobs.n - 1] += 1 << 30;  // the search ends there
  gemm_tn_kernel<kNTile><<<total, kGemmThreads, gemm_smem(kNTile), s>>>(jobs);
  return cudaGetLastError();
}

constexpr int kEwThreads = 256;

__global__ void gather_kernel(const float* __restrict__ x_src, const float* __restrict__ t_src,
                              const int* __restrict__ idx, int n, int bp, int n_in, int in_p,
                              int n_out, int out_p, uint16_t* X, uint16_t* Xt, float* T) {
  const long long e = (long long)blockIdx.x * kEwThreads + threadIdx.x;
  if (e < (long long)bp * in_p) {
    const int r = (int)(e / in_p), c = (int)(e - (e / in_p) * in_p);
    const float v = (r < n && c < n_in) ? x_src[(long long)idx[r] * n_in + c] : 0.f;
    const uint16_t h = f32_to_bf16(v);
    X[(long long)r * in_p + c] = h;
    Xt[(long long)c * bp + r] = h;
  }
  if (t_src && e < (long long)bp * out_p) {
    const int r = (int)(e / out_p), c = (int)(e - (e / out_p) * out_p);
    T[e] = (r < n && c < n_out) ? t_src[(long long)idx[r] * n_out + c] : 0.f;
  }
}

// One warp per sample row: its share of dY in both layouts and its weighted
// squared error.  (One thread summing a row's FP64 errors took 37 us.)
__global__ void loss_grad_kernel(const float* __restrict__ Y, const float* __restrict__ T,
                                 const float* __restrict__ w, int n, int bp, int out_p,
                                 double inv_n, uint16_t* dY, uint16_t* dYt, double* loss_rows) {
  const int r = (int)((blockIdx.x * kEwThreads + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (r >= bp) return;
  double acc = 0.0;
  for (int c = lane; c < out_p; c += 32) {
    const long long e = (long long)r * out_p + c;
    float d = 0.f;
    if (r < n) {
      const double dd = (double)Y[e] - (double)T[e], wc = (double)w[c];
      d = (float)(2.0 * wc * dd * inv_n);
      acc += wc * dd * dd;
    }
    const uint16_t h = f32_to_bf16(d);
    dY[e] = h;
    dYt[(long long)c * bp + r] = h;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0 && r < n) loss_rows[r] = acc;
}

template <typename T>
__device__ __forceinline__ T block_reduce_sum(T v, T* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  T r = 0;
  if (w == 0) {
    r = l < (int)(blockDim.x >> 5) ? sh[l] : (T)0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;  // thread 0
}

__global__ void loss_reduce_kernel(const double* __restrict__ rows, int n, double scale,
                                   double* acc) {
  __shared__ double sh[32];
  double v = 0.0;
  for (int r = threadIdx.x; r < n; r += kEwThreads) v += rows[r];
  v = block_reduce_sum(v, sh);
  if (threadIdx.x == 0) *acc += scale * v;
}

// Adam on every parameter, the bf16 copies of the new weights in both layouts,
// and (the last block) the batch's loss: one launch instead of three and one
// a layer.
__global__ void __launch_bounds__(kEwThreads)
adam_kernel(const __grid_constant__ AdamArgs a) {
  __shared__ double sh[32];
  if (blockIdx.x == gridDim.x - 1) {
    double v = 0.0;
    for (int r = threadIdx.x; r < a.n; r += kEwThreads) v += a.loss_rows[r];
    v = block_reduce_sum(v, sh);
    if (threadIdx.x == 0) *a.loss += a.loss_scale * v;
    return;
  }
  const long long e = (long long)blockIdx.x * kEwThreads + threadIdx.x;
  if (e >= a.count) return;
  const float gg = a.g[e];
  const float mm = fmaf(1.f - a.b1, gg, a.b1 * a.m[e]);
  const float vv = fmaf((1.f - a.b2) * gg, gg, a.b2 * a.v[e]);
  a.m[e] = mm;
  a.v[e] = vv;
  const float p = a.p[e] - a.lr * (mm / a.c1) / (sqrtf(vv / a.c2) + a.eps);
  a.p[e] = p;
  int q = 0;
  while (q + 1 < a.layers && e >= a.woff[q + 1]) q++;
  const long long w = e - a.woff[q];
  const int K = a.K[q], N = a.N[q];
  if (w >= (long long)N * K) return;  // a bias
  const int r = (int)(w / K), c = (int)(w - (w / K) * K);
  const uint16_t h = f32_to_bf16(p);
  a.Wb[q][w] = h;
  a.Wt[q][(long long)c * N + r] = h;
}

__global__ void pack_weights_kernel(const float* __restrict__ W, int N, int K, uint16_t* Wb,
                                    uint16_t* Wt) {
  const long long e = (long long)blockIdx.x * kEwThreads + threadIdx.x;
  if (e >= (long long)N * K) return;
  const int r = (int)(e / K), c = (int)(e - (e / K) * K);
  const uint16_t h = f32_to_bf16(W[e]);
  Wb[e] = h;
  Wt[(long long)c * N + r] = h;
}

inline int ew_blocks(long long count) { return (int)((count + kEwThreads - 1) / kEwThreads); }

}  // namespace

cudaError_t launch_gather(const float* x_src, const float* t_src, const int* idx, int n, int bp,
                          int n_in, int in_p, int n_out, int out_p, uint16_t* X, uint16_t* Xt,
                          float* T, cudaStream_t s) {
  const long long cnt = (long long)bp * (in_p > out_p ? in_p : out_p);
  gather_kernel<<<ew_blocks(cnt), kEwThreads, 0, s>>>(x_src, t_src, idx, n, bp, n_in, in_p,
                                                      n_out, out_p, X, Xt, T);
  return cudaGetLastError();
}

cudaError_t launch_loss_grad(const float* Y, const float* T, const float* w, int n, int bp,
                             int out_p, double inv_n, uint16_t* dY, uint16_t* dYt,
                             double* loss_rows, cudaStream_t s) {
  loss_grad_kernel<<<ew_blocks((long long)bp * 32), kEwThreads, 0, s>>>(
      Y, T, w, n, bp, out_p, inv_n, dY, dYt, loss_rows);
  return cudaGetLastError();
}

cudaError_t launch_loss_reduce(const double* loss_rows, int n, double scale, double* acc,
                               cudaStream_t s) {
  loss_reduce_kernel<<<1, kEwThreads, 0, s>>>(loss_rows, n, scale, acc);
  return cudaGetLastError();
}

cudaError_t launch_adam(AdamArgs a, int t, cudaStream_t s) {
  // bias corrections 1 - beta^t in FP64: in FP32, 1 - 0.999^t loses about
  // nine bits to cancellation at small t
  a.c1 = (float)(1.0 - pow((double)a.b1, (double)t));
  a.c2 = (float)(1.0 - pow((double)a.b2, (double)t));
  adam_kernel<<<ew_blocks(a.count) + 1, kEwThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_pack_weights(const float* W, int N, int K, uint16_t* Wb, uint16_t* Wt,
                                cudaStream_t s) {
  pack_weights_kernel<<<ew_blocks((long long)N * K), kEwThreads, 0, s>>>(W, N, K, Wb, Wt);
  return cudaGetLastError();
}

// Shape rules checked on the host before any launch.
const char* gemm_shape_error(const GemmArgs& g) {
  if (g.M < 1 || g.N < 1 || g.K < 1) return "M, N and K must be >= 1";
  if (g.N > kNMax) return "N must be <= 256";
  if (g.K % 16) return "K must be a multiple of 16";
  if (g.lda < g.K || g.ldb < g.K || g.lda % 8 || g.ldb % 8)
    return "lda and ldb must be >= K and multiples of 8 (16-byte rows)";
  if (((uintptr_t)g.A | (uintptr_t)g.B) & 15) return "A and B must be 16-byte aligned";
  return nullptr;
}

cudaError_t launch_gemms(const GemmArgs* g, int n, cudaStream_t s) {
  GemmJobs jobs{};
  jobs.n = n;
  int wide = 0;
  for (int j = 0; j < n; j++) {
    jobs.g[j] = g[j];
    GemmArgs& x = jobs.g[j];
    const uintptr_t ptrs = (uintptr_t)x.C | (uintptr_t)x.H | (uintptr_t)x.Zin;
    x.vec = !(ptrs & 15) && !(x.ldc % 4) && !(x.ldh % 8) && !(x.ldz % 4);
    if (!x.row_sum) wide += job_ctas(x, kNTileWide);
  }
  // half-width tiles while even those leave the GPU half empty (512 x 256 x 256: 16 CTAs
  // of 64 columns, 32 of 32)
  return wide <= 76 ? launch_jobs<kNTileThin>(jobs, s) : launch_jobs<kNTileWide>(jobs, s);
}

cudaError_t launch_gemm(GemmArgs g, int epi, cudaStream_t s) {
  g.epi = epi;
  return launch_gemms(&g, 1, s);
}

}  // namespace fk

extern "C" fk_status fk_gemm_bf16_tn(const void* A, int64_t lda, const void* B, int64_t ldb,
                                     float* C, int64_t ldc, int32_t M, int32_t N, int32_t K,
                                     int32_t* err_dev, void* cuda_stream) {
  fk::GemmArgs g{};
  g.A = static_cast<const uint16_t*>(A);
  g.B = static_cast<const uint16_t*>(B);
  g.lda = lda;
  g.ldb = ldb;
  g.C = C;
  g.ldc = ldc;
  g.M = M;
  g.N = N;
  g.K = K;
  g.m_valid = M;
  g.err = err_dev;
  if (!A || !B || !C || !err_dev) {
    fk::set_thread_error("fk_gemm_bf16_tn: A, B, C and err must be device pointers");
    return FK_EINVAL;
  }
  if (const char* why = fk::gemm_shape_error(g)) {
    fk::set_thread_error((std::string("fk_gemm_bf16_tn: ") + why).c_str());
    return FK_EINVAL;
  }
  if (ldc < N) {
    fk::set_thread_error("fk_gemm_bf16_tn: ldc must be >= N");
    return FK_EINVAL;
  }
  const cudaError_t e = fk::launch_gemm(g, fk::kEpiF32, static_cast<cudaStream_t>(cuda_stream));
  if (e != cudaSuccess) {
    fk::set_thread_error((std::string("fk_gemm_bf16_tn: ") + cudaGetErrorString(e)).c_str());
    return FK_ECUDA;
  }
  return FK_OK;
}
