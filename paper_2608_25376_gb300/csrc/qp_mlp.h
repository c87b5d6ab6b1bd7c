// Internal interface of the warm-start MLP kernels (qp_mlp.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace qp {
namespace mlp {

enum EpiMode {
  kEpiBiasRelu = 0,   // out_bf16 = bf16(relu(acc + bias))
  kEpiBiasF32 = 1,    // out_f32 = acc + bias
  kEpiPartialF32 = 2, // out_f32 + z * M * ldo = acc for split z (sum_jobs adds them in order)
};

// D[M x N] = A[M x K] B[N x K]^T; A, B bf16 row-major with K contiguous.
// N in [16, 256] and a multiple of 16; K, lda, ldb multiples of 16 / 8.
struct GemmArgs {
  const __nv_bfloat16 *A;
  int lda;
  const __nv_bfloat16 *B;
  int ldb;
  int M, N, K;
  int k_per_split;  // set by gemm()
  int mode;
  const float *bias;
  float *out_f32;
  __nv_bfloat16 *out_bf16;
  int ldo;
  int *err;  // set to 1 if a bounded wait gave up
};

constexpr int kMaxGroup = 4;
// `count` products in one launch, each in the same number of K-splits (their
// tiles run side by side: one product of the weight gradients fills a fifth of
// the SMs).
cudaError_t gemm(const GemmArgs *g, int count, int splits, cudaStream_t st);
// The number of K-splits gemm() launches for K and the requested splits.
int gemm_splits(int K, int splits);
// out[i] = sum over z = 0 .. splits-1, in that order, of ws[z * n + i]: split-K
// partials, or slabs of column sums, added the same way on every run.  Every job
// runs in the same launch, and v's ordered sum into v_sum beside them (v may
// be null): thread j of 256 adds v[j], v[j + 256], ...; then the 256 in order.
struct SumJob {
  const float *ws;
  int splits, n;
  float *out;
};
constexpr int kMaxSums = 8;
cudaError_t sum_jobs(const SumJob *jobs, int count, const float *v, int nv, float *v_sum, cudaStream_t st);

// The network's whole forward pass in one launch, one CTA per 128-row tile:
// x0 bf16 [Mp x 16] (Mp a multiple of 128), weights w[l] bf16 [256 x K_l]
// row-major (K_0 = 16, else 256), bias[l] fp32 [256], hidden activations
// h[l] bf16 [Mp x 256] (null: not written), logits z fp32 [Mp x 256].
struct FwdArgs {
  const __nv_bfloat16 *x0;
  const float *bias[4];
  __nv_bfloat16 *h[3];
  float *z;
  float *z2;  // a second copy of the first rows2 rows of z (null: none; 16-byte aligned)
  int rows2;
  int Mp;
  int *err;  // set to 1 if a bounded wait gave up
};
cudaError_t forward(const FwdArgs &g, const __nv_bfloat16 *const w[4], cudaStream_t st);
// From the logits to the gradients at the hidden activations, in two launches:
// dz bf16 [Mp x 256] = the softmax cross-entropy's
// gradient times inv_rows, loss_rows[m] = -log p[label] of row m (0 for a
// padding row, label < 0), dh[l] bf16 [Mp x 256] = relu'(h[l]) * dY W of the layer
// above.  wt[l]: the transposed weights of layer l (0-based; wt[0] is not read).
struct BwdArgs {
  const float *z;
  const int32_t *label, *steps;
  float inv_rows;
  const __nv_bfloat16 *h[3];
  __nv_bfloat16 *dz, *dh[3];
  float *loss_rows;
  int Mp;
  int *err;  // set to 1 if a bounded wait gave up
};
cudaError_t backward(const BwdArgs &g, const __nv_bfloat16 *const wt[4], cudaStream_t st);
// Column sums of `count` bf16 matrices Y[k] [M x 256], per slab of rows:
// partial + k * kColsumSlabs * 256 gets kColsumSlabs x 256 floats.
constexpr int kColsumSlabs = 64;
cudaError_t colsum(const __nv_bfloat16 *const *Y, int count, int M, float *partial, cudaStream_t st);
// out (cols x rows, row stride rows) = in (rows x cols, contiguous), bf16, for
// every job; cols a multiple of 2, rows a multiple of 64.
struct TransposeJob {
  const __nv_bfloat16 *in;
  __nv_bfloat16 *out;
  int cols;
};
constexpr int kMaxTransposes = 8;
cudaError_t transpose(const TransposeJob *jobs, int count, int rows, cudaStream_t st);

// The parameters in one flat array: W1[256][16], b1[256], then W[256][256],
// b[256] of the other three layers.  wb, wt: the bf16 weights and their
// transposes at the weights' offsets.
constexpr int kParams = 256 * 16 + 256 + 3 * (256 * 256 + 256);
constexpr int weight_offset(int l) { return l == 0 ? 0 : 256 * 16 + 256 + (l - 1) * (256 * 256 + 256); }
constexpr int bias_offset(int l) { return weight_offset(l) + 256 * (l == 0 ? 16 : 256); }
// One Adam step on all of them (Kingma & Ba); nothing happens when *err != 0.
cudaError_t adam(float *w, float *m, float *v, const float *g, float lr, float b1, float b2, float eps, int step,
                 __nv_bfloat16 *wb, __nv_bfloat16 *wt, const int *err, cudaStream_t st);
// wb and wt from the fp32 parameters.
cudaError_t refresh(const float *w, __nv_bfloat16 *wb, __nv_bfloat16 *wt, cudaStream_t st);
// The inputs of a pass: x0 (bf16 [Mp x 16]) from M rows of fp32 features, zero
// rows after them; with labels, their padding rows (label -1, steps 1).
cudaError_t inputs(const float *feats, int M, int Mp, __nv_bfloat16 *x0, int32_t *labels, int32_t *steps,
                   cudaStream_t st);

}  // namespace mlp
}  // namespace qp
