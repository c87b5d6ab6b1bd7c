// Stand-ins for the CUDA runtime, the kernels' launchers and the pointer queries,
// linked with qp_ws.cpp alone: the network's host code runs on the CPU and a test
// sees what it allocates, copies and launches.  "Device" memory is host memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

#include "qp_internal.h"
#include "qp_mlp.h"

namespace {
std::map<void *, size_t> g_allocs;
size_t g_bytes = 0, g_limit = ~size_t(0);
int g_place = qp::kHostMemory;  // where the pointer queries say the caller's buffers are
const void *g_z2 = nullptr;     // of the last forward launch
long g_copied = 0;              // bytes of copies of unspecified direction (to the caller's logits)
std::string g_launches;
std::string g_error;
cudaError_t note(char c) {
  g_launches += c;
  return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_limit(size_t bytes) { g_limit = bytes; }
size_t fake_bytes() { return g_bytes; }
void fake_place(int place) { g_place = place; }
const void *fake_z2() { return g_z2; }
long fake_copied() { return g_copied; }
const char *fake_launches() {
  static std::string out;
  out.swap(g_launches);
  g_launches.clear();
  return out.c_str();
}
const char *fake_error() { return g_error.c_str(); }

cudaError_t cudaFree(void *p) {
  auto it = g_allocs.find(p);
  if (it == g_allocs.end()) std::abort();
  g_bytes -= it->second;
  g_allocs.erase(it);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  if (k == cudaMemcpyDefault) g_copied += (long)n;
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "error"; }
}

namespace qp {
qp_status set_error(qp_status s, const char *msg) {
  g_error = msg;
  return s;
}
bool device_pointer(const void *) { return g_place != kHostMemory; }
int memory_place(const void *) { return g_place; }
bool device_range_fits(const void *, size_t) { return true; }
cudaError_t dev_malloc(void **p, size_t bytes) {
  *p = g_bytes + bytes > g_limit ? nullptr : std::calloc(1, bytes);
  if (!*p) return cudaErrorMemoryAllocation;
  g_allocs[*p] = bytes;
  g_bytes += bytes;
  return cudaSuccess;
}
namespace mlp {
int gemm_splits(int K, int splits) {
  const int kps = ((K + splits - 1) / splits + 63) / 64 * 64;
  return (K + kps - 1) / kps;
}
cudaError_t inputs(const float *, int, int, __nv_bfloat16 *, int32_t *, int32_t *, cudaStream_t) { return note('i'); }
cudaError_t forward(const FwdArgs &g, const __nv_bfloat16 *const *, cudaStream_t) {
  g_z2 = g.z2;
  return note('f');
}
cudaError_t backward(const BwdArgs &, const __nv_bfloat16 *const *, cudaStream_t) { return note('b'); }
cudaError_t gemm(const GemmArgs *, int, int, cudaStream_t) { return note('g'); }
cudaError_t colsum(const __nv_bfloat16 *const *, int, int, float *, cudaStream_t) { return note('c'); }
cudaError_t sum_jobs(const SumJob *, int, const float *, int, float *, cudaStream_t) { return note('s'); }
cudaError_t transpose(const TransposeJob *, int, int, cudaStream_t) { return note('t'); }
cudaError_t refresh(const float *, __nv_bfloat16 *, __nv_bfloat16 *, cudaStream_t) { return note('r'); }
cudaError_t adam(float *, float *, float *, const float *, float, float, float, float, int, __nv_bfloat16 *,
                 __nv_bfloat16 *, const int *, cudaStream_t) {
  return note('a');
}
}  // namespace mlp
}  // namespace qp
