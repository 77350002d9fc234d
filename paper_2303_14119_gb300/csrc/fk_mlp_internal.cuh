// Internal declarations of the surrogate's dense-layer kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fk {

enum GemmEpilogue {
  kEpiF32 = 0,       // C = acc (+ bias)                          FP32 [M][N]
  kEpiBiasGelu = 1,  // C = z = acc + bias (FP32); H = gelu(z) (bf16), Ht = H^T
  kEpiGeluBack = 2,  // H = acc * gelu'(Zin) (bf16), Ht = H^T
};

// C = A * B^T: A [M][lda] and B [N][ldb] bf16 (bit patterns), K-major.
struct GemmArgs {
  const uint16_t* A;
  long long lda;
  const uint16_t* B;
  long long ldb;
  int M, N, K;
  float* C;
  long long ldc;
  const float* bias;  // [N] or null
  uint16_t* H;        // bf16 output [M][ldh]
  long long ldh;
  uint16_t* Ht;       // bf16 transposed output [N][ldht] (or null)
  long long ldht;
  const float* Zin;   // FP32 pre-activation [M][ldz] (kEpiGeluBack)
  long long ldz;
  int m_valid;        // rows >= m_valid write zeros to H / Ht
  int* err;           // set to 1 if a bounded wait ran out
  int epi;            // GemmEpilogue
  int vec;            // 16-byte rows of C, H and Zin (set at the launch)
  // not null: no product, row_sum[r] = sum of the first sum_n values of A's row r
  float* row_sum;
  int sum_n;
};

constexpr int kGemmJobs = 3;
// Independent jobs of one launch.
struct GemmJobs {
  GemmArgs g[kGemmJobs];
  int ctas[kGemmJobs];
  int n;
};

constexpr int kMaxLayers = 33;
struct AdamArgs {
  float *p, *m, *v;
  const float* g;
  long long count;
  float lr, b1, b2, eps, c1, c2;
  // the layers' weights in the parameter vector, and their bf16 copies [N][K], [K][N]
  int layers;
  int K[kMaxLayers], N[kMaxLayers];
  long long woff[kMaxLayers];
  uint16_t *Wb[kMaxLayers], *Wt[kMaxLayers];
  // *loss += loss_scale * sum of loss_rows[0 .. n)
  const double* loss_rows;
  int n;
  double loss_scale;
  double* loss;
};

// Elementwise and reduction kernels of training and inference.
// Rows [0, n) of the gathered batch come from samples idx[r] of the data
// set (FP32 [*][n_in]); rows >= n are zero.  X [bp][in_p] and its
// transpose Xt [in_p][bp] in bf16; T [bp][out_p] FP32 (when t_src is set).
cudaError_t launch_gather(const float* x_src, const float* t_src, const int* idx, int n, int bp,
                          int n_in, int in_p, int n_out, int out_p, uint16_t* X, uint16_t* Xt,
                          float* T, cudaStream_t s);
// dY = 2 w (Y - T) / n_total for rows < n (bf16, both layouts), zero
// elsewhere; loss_rows[r] = sum_o w_o (Y - T)^2 (FP64, rows < n).
cudaError_t launch_loss_grad(const float* Y, const float* T, const float* w, int n, int bp,
                             int out_p, double inv_n, uint16_t* dY, uint16_t* dYt,
                             double* loss_rows, cudaStream_t s);
// *acc += scale * sum_{r < n} loss_rows[r] (one block, fixed order)
cudaError_t launch_loss_reduce(const double* loss_rows, int n, double scale, double* acc,
                               cudaStream_t s);
// Adam (bias-corrected step t >= 1; c1 and c2 are set here), the bf16 weights
// and the batch's loss.
cudaError_t launch_adam(AdamArgs a, int t, cudaStream_t s);
// bf16 copies of a layer's FP32 weights W [N][K]: Wb [N][K] and Wt [K][N]
cudaError_t launch_pack_weights(const float* W, int N, int K, uint16_t* Wb, uint16_t* Wt,
                                cudaStream_t s);

// nullptr if the shape is supported, else the reason
const char* gemm_shape_error(const GemmArgs& g);
cudaError_t launch_gemm(GemmArgs g, int epi, cudaStream_t s);
// n <= kGemmJobs independent jobs in one launch (epi of each set)
cudaError_t launch_gemms(const GemmArgs* g, int n, cudaStream_t s);

}  // namespace fk
