// Host side of the learned warm start: per-cell features of a field, the MLP
// (16 -> 256 -> 256 -> 256 -> 256 step logits, bf16 weights with fp32 masters
// and Adam moments), its forward pass, one training step (forward, softmax
// cross-entropy, backward, Adam) built from the tcgen05 GEMM and the small
// kernels of qp_mlp.cu, and the greedy decode of step logits into a feasible
// one-hot state.  The public contract is in include/qpath.h.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <utility>
#include <vector>

#include "qp_internal.h"
#include "qp_mlp.h"

using namespace qp;

namespace {

constexpr int kIn = 16, kHid = 256, kOut = 256;
constexpr int kLayers = 4;
const int kDimIn[kLayers] = {kIn, kHid, kHid, kHid};
const int kDimOut[kLayers] = {kHid, kHid, kHid, kOut};

struct Buf {
  void *p = nullptr;
  size_t bytes = 0;
  ~Buf() {
    if (p) cudaFree(p);
  }
  bool ensure(size_t want) {
    if (want <= bytes) return true;
    if (p) cudaFree(p);
    p = nullptr;
    bytes = 0;
    if (dev_malloc(&p, want) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
      return false;
    }
    bytes = want;
    return true;
  }
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    bytes = 0;
  }
  template <typename T>
  T *as() const { return static_cast<T *>(p); }
};

#define WS_CU(call)                                                                   \
  do {                                                                                \
    cudaError_t e_ = (call);                                                          \
    if (e_ != cudaSuccess) return set_error(QP_ECUDA, cudaGetErrorString(e_));        \
  } while (0)
#define WS_ALLOC(buf, bytes)                                                          \
  do {                                                                                \
    if (!(buf).ensure(bytes)) return set_error(QP_ENOMEM, "warm start: cudaMalloc failed"); \
  } while (0)

uint64_t splitmix64(uint64_t &s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

// What a call reads back when it ends: the tensor-core waits' flag and the sum
// of the rows' losses.
struct PassResult {
  int err;
  float loss;
};

struct qp_ws {
  int dev = 0;
  int step = 0;
  Buf par, am, av, grad;               // fp32 masters, Adam's moments, gradients: flat (mlp::kParams)
  Buf wb, wt;                          // bf16 weights and their transposes, at the weights' flat offsets
  int cap = 0;                         // rows of the largest pass so far
  int fwd_mode = QP_WS_FORWARD_FUSED;
  Buf x0, z, res;                      // z holds the fp32 features until they are converted
  Buf h[3];                            // passes that keep the hidden activations
  Buf dz, dh[3], lab, stp;             // training passes, as the rest
  Buf tr;              // transposes for the weight gradients: dY and X of `group` layers
  Buf gws, cws, lrow;  // split-K partials of `group` layers, column-sum partials, per-row losses (fixed-order sums)
  int group = 0;       // layers whose weight gradients are computed side by side: all, or 1 when memory is short

  float *weight(const Buf &b, int l) const { return b.as<float>() + mlp::weight_offset(l); }
  float *bias(const Buf &b, int l) const { return b.as<float>() + mlp::bias_offset(l); }
  __nv_bfloat16 *weight16(const Buf &b, int l) const { return b.as<__nv_bfloat16>() + mlp::weight_offset(l); }
  PassResult *result() const { return res.as<PassResult>(); }
};

namespace {

static_assert(kIn == 16 && kHid == 256 && kOut == 256 && kLayers == 4, "the flat layout of mlp::kParams");

int weight_splits(int Mp) { return std::max(1, Mp / 512); }

// The buffers of a pass over Mp rows.  A row takes 1056 bytes, 2592 with the
// hidden activations and 8268 in training; where those cannot be had, the weight
// gradients of the layers share one layer's buffers and it is 5676.
qp_status ensure_rows(qp_ws *m, int Mp, bool hidden, bool train) {
  const int cap = m->cap;
  if (Mp > cap) m->cap = 0;  // until the growth below has succeeded
  const size_t rows = Mp;
  WS_ALLOC(m->x0, rows * kIn * 2);
  WS_ALLOC(m->z, rows * kOut * 4);
  if (hidden)
    for (int i = 0; i < 3; ++i) WS_ALLOC(m->h[i], rows * kHid * 2);
  if (train) {
    for (int i = 0; i < 3; ++i) WS_ALLOC(m->dh[i], rows * kHid * 2);
    WS_ALLOC(m->dz, rows * kOut * 2);
    WS_ALLOC(m->lab, rows * 4);
    WS_ALLOC(m->stp, rows * 4);
    WS_ALLOC(m->lrow, rows * 4);
    WS_ALLOC(m->cws, (size_t)kLayers * mlp::kColsumSlabs * kOut * 4);
    const size_t zs = mlp::gemm_splits(Mp, weight_splits(Mp));
    m->group = kLayers;
    if (!m->tr.ensure(rows * (kLayers * kHid + kIn + 3 * kHid) * 2) || !m->gws.ensure(zs * mlp::kParams * 4)) {
      m->group = 1;
      m->tr.release();
      m->gws.release();
      WS_ALLOC(m->tr, rows * 2 * kHid * 2);
      WS_ALLOC(m->gws, zs * kHid * kHid * 4);
    }
  }
  m->cap = std::max(cap, Mp);
  return QP_OK;
}

// The pass's inputs to the device; the features become bf16 there (converting
// them on the host took 60 us of a 16384-cell pass).  The copies may still be
// reading the caller's buffers on return: every caller waits for the stream.
qp_status upload_inputs(qp_ws *m, const float *feats, int M, int Mp, const int32_t *labels, const int32_t *steps,
                        cudaStream_t st) {
  const bool train = labels && steps;
  if (qp_status s = ensure_rows(m, Mp, train || m->fwd_mode != QP_WS_FORWARD_FUSED, train); s != QP_OK) return s;
  WS_CU(cudaMemcpyAsync(m->z.p, feats, (size_t)M * kIn * 4, cudaMemcpyHostToDevice, st));
  if (train) {
    WS_CU(cudaMemcpyAsync(m->lab.p, labels, (size_t)M * 4, cudaMemcpyHostToDevice, st));
    WS_CU(cudaMemcpyAsync(m->stp.p, steps, (size_t)M * 4, cudaMemcpyHostToDevice, st));
  }
  WS_CU(mlp::inputs(m->z.as<float>(), M, Mp, m->x0.as<__nv_bfloat16>(), train ? m->lab.as<int32_t>() : nullptr,
                    train ? m->stp.as<int32_t>() : nullptr, st));
  return QP_OK;
}

mlp::GemmArgs gargs(const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B, int ldb, int M, int N, int K,
                    int mode, int *err) {
  mlp::GemmArgs g{};
  g.A = A; g.lda = lda; g.B = B; g.ldb = ldb; g.M = M; g.N = N; g.K = K; g.mode = mode; g.err = err;
  return g;
}

// Logits into m->z (and their first rows into out, when given: device memory,
// 16-byte aligned, fused mode); the hidden activations into m->h[] when
// keep_hidden (the backward pass reads them) or when the layers run as separate
// launches.
qp_status forward(qp_ws *m, int Mp, bool keep_hidden, float *out, int rows, cudaStream_t st) {
  int *err = &m->result()->err;
  if (m->fwd_mode == QP_WS_FORWARD_FUSED) {
    mlp::FwdArgs g{};
    g.x0 = m->x0.as<__nv_bfloat16>();
    const __nv_bfloat16 *w[kLayers];
    for (int l = 0; l < kLayers; ++l) {
      g.bias[l] = m->bias(m->par, l);
      w[l] = m->weight16(m->wb, l);
    }
    for (int l = 0; l < 3; ++l) g.h[l] = keep_hidden ? m->h[l].as<__nv_bfloat16>() : nullptr;
    g.z = m->z.as<float>();
    g.z2 = out;
    g.rows2 = rows;
    g.Mp = Mp;
    g.err = err;
    WS_CU(mlp::forward(g, w, st));
    return QP_OK;
  }
  const __nv_bfloat16 *in = m->x0.as<__nv_bfloat16>();
  int ldin = kIn;
  for (int l = 0; l < kLayers; ++l) {
    mlp::GemmArgs g = gargs(in, ldin, m->weight16(m->wb, l), kDimIn[l], Mp, kDimOut[l], kDimIn[l],
                            l < 3 ? mlp::kEpiBiasRelu : mlp::kEpiBiasF32, err);
    g.bias = m->bias(m->par, l);
    if (l < 3) {
      g.out_bf16 = m->h[l].as<__nv_bfloat16>();
      g.ldo = kHid;
    } else {
      g.out_f32 = m->z.as<float>();
      g.ldo = kOut;
    }
    WS_CU(mlp::gemm(&g, 1, 1, st));
    in = m->h[l < 3 ? l : 2].as<__nv_bfloat16>();
    ldin = kHid;
  }
  return QP_OK;
}

// Gradients of the mean cross-entropy into m->grad; the loss sum into m->res.
// Every sum over rows is taken in a fixed order (split-K partials and slabs
// added in index order, no atomics), so a training run repeats bit for bit.
// The chain of the dX products runs in one launch, and everything else of the
// four layers side by side in one launch of its kind (of one layer after the
// other when the buffers are shared: the same products and sums).
qp_status backward(qp_ws *m, int M, int Mp, cudaStream_t st) {
  int *err = &m->result()->err;
  mlp::BwdArgs bw{};
  bw.z = m->z.as<float>();
  bw.label = m->lab.as<int32_t>();
  bw.steps = m->stp.as<int32_t>();
  bw.inv_rows = 1.0f / (float)M;
  bw.dz = m->dz.as<__nv_bfloat16>();
  bw.loss_rows = m->lrow.as<float>();
  bw.Mp = Mp;
  bw.err = err;
  const __nv_bfloat16 *wt[kLayers];
  for (int l = 0; l < kLayers; ++l) wt[l] = m->weight16(m->wt, l);
  for (int l = 0; l < 3; ++l) {
    bw.h[l] = m->h[l].as<__nv_bfloat16>();
    bw.dh[l] = m->dh[l].as<__nv_bfloat16>();
  }
  WS_CU(mlp::backward(bw, wt, st));
  const int splits = weight_splits(Mp), zs = mlp::gemm_splits(Mp, splits);
  const __nv_bfloat16 *dy[kLayers], *x[kLayers];
  for (int l = 0; l < kLayers; ++l) {
    dy[l] = l == kLayers - 1 ? m->dz.as<__nv_bfloat16>() : m->dh[l].as<__nv_bfloat16>();
    x[l] = l == 0 ? m->x0.as<__nv_bfloat16>() : m->h[l - 1].as<__nv_bfloat16>();
  }
  // dW[out][in] = sum_m dY[m][out] X[m][in]  (operands transposed so m is contiguous)
  for (int l0 = 0; l0 < kLayers; l0 += m->group) {
    __nv_bfloat16 *tr = m->tr.as<__nv_bfloat16>();
    mlp::TransposeJob tj[2 * kLayers];
    mlp::GemmArgs g[kLayers];
    mlp::SumJob sums[2 * kLayers];
    float *ws = m->gws.as<float>();
    for (int k = 0; k < m->group; ++k) {
      const int l = l0 + k;
      __nv_bfloat16 *dyt = tr, *xt = tr + (size_t)Mp * kDimOut[l];
      tr = xt + (size_t)Mp * kDimIn[l];
      tj[2 * k] = {dy[l], dyt, kDimOut[l]};
      tj[2 * k + 1] = {x[l], xt, kDimIn[l]};
      g[k] = gargs(dyt, Mp, xt, Mp, kDimOut[l], kDimIn[l], Mp, mlp::kEpiPartialF32, err);
      g[k].out_f32 = ws;
      g[k].ldo = kDimIn[l];
      const int n = kDimOut[l] * kDimIn[l];
      sums[2 * k] = {ws, zs, n, m->weight(m->grad, l)};
      sums[2 * k + 1] = {m->cws.as<float>() + (size_t)l * mlp::kColsumSlabs * kOut, mlp::kColsumSlabs, kOut,
                         m->bias(m->grad, l)};
      ws += (size_t)zs * n;
    }
    WS_CU(mlp::transpose(tj, 2 * m->group, Mp, st));
    WS_CU(mlp::gemm(g, m->group, splits, st));
    if (l0 == 0) WS_CU(mlp::colsum(dy, kLayers, Mp, m->cws.as<float>(), st));
    WS_CU(mlp::sum_jobs(sums, 2 * m->group, l0 == 0 ? m->lrow.as<float>() : nullptr, Mp, &m->result()->loss, st));
  }
  return QP_OK;
}

// Wait for the pass and read its result (and, into grads_out when given, the gradients).
qp_status finish(qp_ws *m, float *grads_out, PassResult *out, cudaStream_t st) {
  if (grads_out) WS_CU(cudaMemcpyAsync(grads_out, m->grad.p, (size_t)mlp::kParams * 4, cudaMemcpyDeviceToHost, st));
  WS_CU(cudaMemcpyAsync(out, m->res.p, sizeof *out, cudaMemcpyDeviceToHost, st));
  WS_CU(cudaStreamSynchronize(st));
  if (out->err) {
    WS_CU(cudaMemsetAsync(&m->result()->err, 0, 4, st));
    return set_error(QP_ETIMEOUT, "warm start: a tensor-core wait gave up");
  }
  return QP_OK;
}

// A failed call leaves no copy reading the caller's buffers.
qp_status settle(qp_status s, cudaStream_t st) {
  if (s != QP_OK && cudaStreamSynchronize(st) != cudaSuccess) cudaGetLastError();
  return s;
}

struct DevGuard {
  int prev = -1;
  explicit DevGuard(int dev) {
    int cur = 0;
    if (cudaGetDevice(&cur) == cudaSuccess && cur != dev) {
      prev = cur;
      cudaSetDevice(dev);
    }
  }
  ~DevGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

}  // namespace

extern "C" qp_status qp_ws_create(uint64_t seed, qp_ws **out) {
  if (!out) return set_error(QP_EINVAL, "out is NULL");
  *out = nullptr;
  auto m = std::make_unique<qp_ws>();
  if (cudaGetDevice(&m->dev) != cudaSuccess) return set_error(QP_ECUDA, "cudaGetDevice failed");
  const size_t n = mlp::kParams;
  if (!m->par.ensure(n * 4) || !m->am.ensure(n * 4) || !m->av.ensure(n * 4) || !m->grad.ensure(n * 4) ||
      !m->wb.ensure(n * 2) || !m->wt.ensure(n * 2) || !m->res.ensure(sizeof(PassResult)))
    return set_error(QP_ENOMEM, "warm start: cudaMalloc failed");
  // He-uniform initialisation from a splitmix64 stream, zero biases
  std::vector<float> p(n, 0.0f);
  uint64_t s = seed;
  for (int l = 0; l < kLayers; ++l) {
    const double lim = std::sqrt(6.0 / kDimIn[l]);
    float *w = p.data() + mlp::weight_offset(l);
    for (int e = 0; e < kDimOut[l] * kDimIn[l]; ++e) {
      const double u = (double)(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0);
      w[e] = (float)((2.0 * u - 1.0) * lim);
    }
  }
  WS_CU(cudaMemset(m->am.p, 0, n * 4));
  WS_CU(cudaMemset(m->av.p, 0, n * 4));
  WS_CU(cudaMemset(m->res.p, 0, sizeof(PassResult)));
  WS_CU(cudaMemcpy(m->par.p, p.data(), n * 4, cudaMemcpyHostToDevice));
  WS_CU(mlp::refresh(m->par.as<float>(), m->wb.as<__nv_bfloat16>(), m->wt.as<__nv_bfloat16>(), nullptr));
  WS_CU(cudaStreamSynchronize(nullptr));
  *out = m.release();
  return QP_OK;
}

extern "C" void qp_ws_destroy(qp_ws *m) {
  if (!m) return;
  DevGuard g(m->dev);
  delete m;
}

extern "C" int64_t qp_ws_param_count(void) { return mlp::kParams; }

extern "C" qp_status qp_ws_get_params(qp_ws *m, float *out) {
  if (!m || !out) return set_error(QP_EINVAL, "NULL argument");
  DevGuard g(m->dev);
  WS_CU(cudaMemcpy(out, m->par.p, (size_t)mlp::kParams * 4, cudaMemcpyDeviceToHost));
  return QP_OK;
}

extern "C" qp_status qp_ws_set_params(qp_ws *m, const float *in) {
  if (!m || !in) return set_error(QP_EINVAL, "NULL argument");
  DevGuard g(m->dev);
  WS_CU(cudaMemcpy(m->par.p, in, (size_t)mlp::kParams * 4, cudaMemcpyHostToDevice));
  WS_CU(mlp::refresh(m->par.as<float>(), m->wb.as<__nv_bfloat16>(), m->wt.as<__nv_bfloat16>(), nullptr));
  WS_CU(cudaStreamSynchronize(nullptr));
  return QP_OK;
}

extern "C" qp_status qp_ws_forward(qp_ws *m, const float *feats, int32_t M, float *logits_out, void *stream) {
  if (!m || !feats || !logits_out || M < 1) return set_error(QP_EINVAL, "bad argument");
  const int place = memory_place(logits_out);
  if (place != kHostMemory && !device_range_fits(logits_out, (size_t)M * kOut * 4))
    return set_error(QP_EINVAL, "qp_ws_forward: the device buffer for the logits is too small");
  DevGuard g(m->dev);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int Mp = (M + 127) / 128 * 128;
  // the fused kernel writes the caller's logits beside its own when they lie on its GPU (another GPU's memory need not
  // be mapped here: those are copied)
  const bool direct =
      place == m->dev && m->fwd_mode == QP_WS_FORWARD_FUSED && (reinterpret_cast<uintptr_t>(logits_out) & 15) == 0;
  PassResult r{};
  const auto pass = [&]() -> qp_status {
    if (qp_status s = upload_inputs(m, feats, M, Mp, nullptr, nullptr, st); s != QP_OK) return s;
    if (qp_status s = forward(m, Mp, false, direct ? logits_out : nullptr, M, st); s != QP_OK) return s;
    if (!direct) WS_CU(cudaMemcpyAsync(logits_out, m->z.p, (size_t)M * kOut * 4, cudaMemcpyDefault, st));
    return finish(m, nullptr, &r, st);
  };
  return settle(pass(), st);
}

extern "C" qp_status qp_ws_set_forward_mode(qp_ws *m, int32_t mode) {
  if (!m || (mode != QP_WS_FORWARD_FUSED && mode != QP_WS_FORWARD_LAYERED))
    return set_error(QP_EINVAL, "bad argument");
  m->fwd_mode = mode;
  return QP_OK;
}

extern "C" qp_status qp_ws_grads(qp_ws *m, const float *feats, const int32_t *labels, const int32_t *steps,
                                 int32_t M, float *grads_out, float *loss_out, void *stream) {
  if (!m || !feats || !labels || !steps || M < 1) return set_error(QP_EINVAL, "bad argument");
  DevGuard g(m->dev);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int Mp = (M + 127) / 128 * 128;
  PassResult r{};
  const auto pass = [&]() -> qp_status {
    if (qp_status s = upload_inputs(m, feats, M, Mp, labels, steps, st); s != QP_OK) return s;
    if (qp_status s = forward(m, Mp, true, nullptr, 0, st); s != QP_OK) return s;
    if (qp_status s = backward(m, M, Mp, st); s != QP_OK) return s;
    return finish(m, grads_out, &r, st);
  };
  if (qp_status s = settle(pass(), st); s != QP_OK) return s;
  if (loss_out) *loss_out = r.loss / (float)M;
  return QP_OK;
}

extern "C" qp_status qp_ws_train_step(qp_ws *m, const float *feats, const int32_t *labels, const int32_t *steps,
                                      int32_t M, float lr, float *loss_out, void *stream) {
  if (!m || !feats || !labels || !steps || M < 1) return set_error(QP_EINVAL, "bad argument");
  DevGuard g(m->dev);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int Mp = (M + 127) / 128 * 128;
  PassResult r{};
  const auto pass = [&]() -> qp_status {
    if (qp_status s = upload_inputs(m, feats, M, Mp, labels, steps, st); s != QP_OK) return s;
    if (qp_status s = forward(m, Mp, true, nullptr, 0, st); s != QP_OK) return s;
    if (qp_status s = backward(m, M, Mp, st); s != QP_OK) return s;
    // the update reads the pass's error flag on the device and leaves a failed pass's parameters alone
    WS_CU(mlp::adam(m->par.as<float>(), m->am.as<float>(), m->av.as<float>(), m->grad.as<float>(), lr, 0.9f, 0.999f,
                    1e-8f, m->step + 1, m->wb.as<__nv_bfloat16>(), m->wt.as<__nv_bfloat16>(), &m->result()->err, st));
    return finish(m, nullptr, &r, st);
  };
  if (qp_status s = settle(pass(), st); s != QP_OK) return s;
  m->step += 1;
  if (loss_out) *loss_out = r.loss / (float)M;
  return QP_OK;
}

// ----------------------------------------------------------------------------- read-back
extern "C" qp_status qp_ws_get_state(qp_ws *m, int32_t which, float *out) {
  if (!m || !out || which < QP_WS_STATE_PARAMS || which > QP_WS_STATE_GRADS)
    return set_error(QP_EINVAL, "bad argument");
  DevGuard g(m->dev);
  WS_CU(cudaDeviceSynchronize());
  const Buf &b = which == QP_WS_STATE_PARAMS ? m->par
                 : which == QP_WS_STATE_ADAM_M ? m->am
                 : which == QP_WS_STATE_ADAM_V ? m->av : m->grad;
  WS_CU(cudaMemcpy(out, b.p, (size_t)mlp::kParams * 4, cudaMemcpyDeviceToHost));
  return QP_OK;
}

extern "C" qp_status qp_ws_get_buffer(qp_ws *m, int32_t which, int32_t rows, void *out) {
  if (!m || !out) return set_error(QP_EINVAL, "bad argument");
  DevGuard g(m->dev);
  for (const auto &w : {std::make_pair((int)QP_WS_BUF_W_BF16, &m->wb), std::make_pair((int)QP_WS_BUF_WT_BF16, &m->wt)})
    if (which >= w.first && which < w.first + kLayers) {
      const int l = which - w.first;
      WS_CU(cudaDeviceSynchronize());
      WS_CU(cudaMemcpy(out, m->weight16(*w.second, l), (size_t)kDimOut[l] * kDimIn[l] * 2, cudaMemcpyDeviceToHost));
      return QP_OK;
    }
  if (rows < 1 || rows > m->cap) return set_error(QP_EINVAL, "rows beyond the last pass's buffers");
  Buf *b = nullptr;
  size_t row_bytes = (size_t)kHid * 2;
  switch (which) {
    case QP_WS_BUF_X0: b = &m->x0; row_bytes = (size_t)kIn * 2; break;
    case QP_WS_BUF_H1: case QP_WS_BUF_H2: case QP_WS_BUF_H3: b = &m->h[which - QP_WS_BUF_H1]; break;
    case QP_WS_BUF_Z: b = &m->z; row_bytes = (size_t)kOut * 4; break;
    case QP_WS_BUF_DZ: b = &m->dz; row_bytes = (size_t)kOut * 2; break;
    case QP_WS_BUF_DH1: case QP_WS_BUF_DH2: case QP_WS_BUF_DH3: b = &m->dh[which - QP_WS_BUF_DH1]; break;
    default: return set_error(QP_EINVAL, "unknown buffer");
  }
  WS_CU(cudaDeviceSynchronize());
  WS_ALLOC(*b, (size_t)rows * row_bytes);  // no pass has written it: no defined values
  WS_CU(cudaMemcpy(out, b->p, (size_t)rows * row_bytes, cudaMemcpyDeviceToHost));
  return QP_OK;
}

// ----------------------------------------------------------------------------- features
extern "C" qp_status qp_ws_features(const qp_field *f, float *feats_out, int32_t *n_cells) {
  if (!f || f->rows < 1 || f->cols < 1) return set_error(QP_EINVAL, "bad field");
  const int H = f->rows, W = f->cols;
  auto isfree = [&](int r, int c) {
    if (r < 0 || r >= H || c < 0 || c >= W) return false;
    return !f->free_mask || f->free_mask[r * W + c] != 0;
  };
  if (f->start < 0 || f->start >= H * W || !isfree(f->start / W, f->start % W))
    return set_error(QP_EINVAL, "start cell is not a free cell of the grid");
  const int rs = f->start / W, cs = f->start % W;
  int C = 0;
  for (int r = 0; r < H; ++r)
    for (int c = 0; c < W; ++c) C += isfree(r, c);
  if (n_cells) *n_cells = C;
  if (!feats_out) return QP_OK;
  int k = 0;
  for (int r = 0; r < H; ++r)
    for (int c = 0; c < W; ++c) {
      if (!isfree(r, c)) continue;
      int blocked8 = 0, free25 = 0;
      for (int dr = -2; dr <= 2; ++dr)
        for (int dc = -2; dc <= 2; ++dc) {
          const bool fr = isfree(r + dr, c + dc);
          free25 += fr;
          if (std::abs(dr) <= 1 && std::abs(dc) <= 1 && (dr || dc)) blocked8 += !fr;
        }
      float *x = feats_out + (size_t)k * kIn;
      x[0] = c / 15.0f;                        // x
      x[1] = r / 15.0f;                        // y
      x[2] = blocked8 / 8.0f;                  // obstacle context: blocked or outside among the 8 neighbours
      x[3] = cs / 15.0f;
      x[4] = rs / 15.0f;
      x[5] = W / 16.0f;
      x[6] = H / 16.0f;
      x[7] = C / 256.0f;
      x[8] = (c - cs) / 15.0f;
      x[9] = (r - rs) / 15.0f;
      x[10] = W > 1 ? c / (float)(W - 1) : 0.0f;
      x[11] = H > 1 ? r / (float)(H - 1) : 0.0f;
      x[12] = free25 / 25.0f;
      x[13] = (float)(r & 1);
      x[14] = 1.0f;
      x[15] = 0.0f;
      ++k;
    }
  return QP_OK;
}

// ----------------------------------------------------------------------------- decode
extern "C" qp_status qp_ws_decode(const float *logits, int32_t ld, int32_t C, int32_t start_cell, uint8_t *state_out,
                                  int32_t *path_out) {
  if (!logits || C < 1 || C > kOut || start_cell < 0 || start_cell >= C || ld < C)
    return set_error(QP_EINVAL, "bad argument");
  // Greedy matching: the start cell takes step 0; then repeatedly the largest
  // logit among unassigned cells and free steps 1..C-1 fixes one (cell, step)
  // pair (ties: smaller cell, then smaller step).  Each unassigned cell keeps
  // its best free step; only cells whose best step was just taken rescan.
  std::vector<int32_t> path(C, -1), best(C, -1);
  std::vector<char> cell_done(C, 0), step_done(C, 0);
  path[0] = start_cell;
  cell_done[start_cell] = 1;
  step_done[0] = 1;
  auto rescan = [&](int i) {
    int bt = -1;
    float bv = 0.0f;
    for (int t = 1; t < C; ++t) {
      if (step_done[t]) continue;
      const float v = logits[(size_t)i * ld + t];
      if (bt < 0 || v > bv) {
        bt = t;
        bv = v;
      }
    }
    best[i] = bt;
  };
  for (int i = 0; i < C; ++i)
    if (!cell_done[i]) rescan(i);
  for (int round = 1; round < C; ++round) {
    int bi = -1;
    float bv = 0.0f;
    for (int i = 0; i < C; ++i) {
      if (cell_done[i]) continue;
      const float v = logits[(size_t)i * ld + best[i]];
      if (bi < 0 || v > bv || (v == bv && i < bi)) {
        bi = i;
        bv = v;
      }
    }
    const int t = best[bi];
    path[t] = bi;
    cell_done[bi] = 1;
    step_done[t] = 1;
    for (int i = 0; i < C; ++i)
      if (!cell_done[i] && best[i] == t) rescan(i);
  }
  if (state_out) {
    std::memset(state_out, 0, (size_t)C * C);
    for (int t = 0; t < C; ++t) state_out[(size_t)t * C + path[t]] = 1;
  }
  if (path_out) std::memcpy(path_out, path.data(), (size_t)C * 4);
  return QP_OK;
}

// A walk guided by the predicted steps: from the start cell, move each step to
// the unvisited cell nearest to the current one (distance matrix d), choosing
// among equally near cells the one with the smallest expected step
// E_j = sum_t softmax(logits_j)_t * t over t < C (then the smaller cell id).
extern "C" qp_status qp_ws_decode_walk(const float *logits, int32_t ld, int32_t C, int32_t start_cell,
                                       const int32_t *d, uint8_t *state_out, int32_t *path_out) {
  if (!logits || !d || C < 1 || C > kOut || start_cell < 0 || start_cell >= C || ld < C)
    return set_error(QP_EINVAL, "bad argument");
  std::vector<double> e(C);
  for (int i = 0; i < C; ++i) {
    const float *z = logits + (size_t)i * ld;
    double mx = z[0];
    for (int t = 1; t < C; ++t) mx = std::max(mx, (double)z[t]);
    double s = 0.0, st = 0.0;
    for (int t = 0; t < C; ++t) {
      const double p = std::exp((double)z[t] - mx);
      s += p;
      st += p * t;
    }
    e[i] = st / s;
  }
  std::vector<int32_t> path(C);
  std::vector<char> seen(C, 0);
  int cur = start_cell;
  path[0] = cur;
  seen[cur] = 1;
  for (int t = 1; t < C; ++t) {
    int nb = -1;
    for (int j = 0; j < C; ++j) {
      if (seen[j]) continue;
      if (nb < 0) {
        nb = j;
        continue;
      }
      const int32_t dj = d[(size_t)cur * C + j], db = d[(size_t)cur * C + nb];
      if (dj < db || (dj == db && e[j] < e[nb])) nb = j;
    }
    path[t] = nb;
    seen[nb] = 1;
    cur = nb;
  }
  if (state_out) {
    std::memset(state_out, 0, (size_t)C * C);
    for (int t = 0; t < C; ++t) state_out[(size_t)t * C + path[t]] = 1;
  }
  if (path_out) std::memcpy(path_out, path.data(), (size_t)C * 4);
  return QP_OK;
}

// ----------------------------------------------------------------------------- one-call inference
extern "C" qp_status qp_ws_infer(qp_ws *m, const qp_field *field, const int32_t *d, uint8_t *state_out,
                                 int32_t *path_out, void *stream) {
  if (!m || !field || (!state_out && !path_out)) return set_error(QP_EINVAL, "bad argument");
  int32_t C = 0;
  qp_status s = qp_ws_features(field, nullptr, &C);
  if (s != QP_OK) return s;
  if (C < 1 || C > kOut) return set_error(QP_ERANGE, "the field has more cells than the network has steps");
  std::vector<float> feats((size_t)C * kIn), logits((size_t)C * kOut);
  s = qp_ws_features(field, feats.data(), nullptr);
  if (s != QP_OK) return s;
  s = qp_ws_forward(m, feats.data(), C, logits.data(), stream);
  if (s != QP_OK) return s;
  // the start cell's id: free cells before it in row-major order
  int start = 0;
  for (int g = 0; g < field->start; ++g) start += !field->free_mask || field->free_mask[g] != 0;
  return d ? qp_ws_decode_walk(logits.data(), kOut, C, start, d, state_out, path_out)
           : qp_ws_decode(logits.data(), kOut, C, start, state_out, path_out);
}
