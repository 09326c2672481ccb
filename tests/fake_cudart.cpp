// The host API (csrc/mr_api.cu) over a stand-in for the CUDA runtime: "device" memory
// is the host's, kernels do nothing, and one chosen runtime call fails.  Linked and run
// by tests/test_host_errors.py, without a GPU.  For every runtime call of mr_cnn_eval in
// turn it prints the call's name, the status of mr_cnn_eval when that call fails, and
// the copies from or to the caller's arrays still queued when it returned.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "mr_cnn.h"

namespace {
int calls = 0, fail_at = 0, queued = 0;
const char* name = "";
cudaError_t call(const char* n) {
  if (++calls != fail_at) return cudaSuccess;
  name = n;
  return cudaErrorUnknown;
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  p->multiProcessorCount = 4;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "chosen failure"; }
cudaError_t cudaGetLastError() { return call("cudaGetLastError"); }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  const cudaError_t e = call("cudaMallocAsync");
  if (e == cudaSuccess) *p = std::calloc(n, 1);
  return e;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  const cudaError_t e = call("cudaMemcpyAsync");
  if (e != cudaSuccess) return e;
  std::memcpy(d, s, n);
  ++queued;  // pinned memory: the copy may run until the stream is waited for
  return e;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  const cudaError_t e = call("cudaMemsetAsync");
  if (e == cudaSuccess) std::memset(d, v, n);
  return e;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  const cudaError_t e = call("cudaStreamSynchronize");
  if (e == cudaSuccess) queued = 0;
  return e;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}

namespace mr {
// kernels whose addresses the host API takes, and the launchers on this path
void k_step_begin(Counters*, int32_t*) {}
void k_time_coef(TreeTime*, const TreeDev*, int, int) {}
void k_time_advance(TreeTime*, int) {}
int cnn_tile(int Bs) { return Bs + 2 * kG; }
void launch_train(int, const float*, const float*, const int32_t*, int64_t, int, const float*, float, float*, float*,
                  float*, int, cudaStream_t) {}
}  // namespace mr

int main() {
  mr_params p{};
  p.dim = 2; p.Bs = 17; p.ng = 4; p.nvar = 1; p.ntrees = 1; p.precision = MR_PREC_FP32; p.rhs_kind = MR_RHS_ADV;
  p.L = 1.0; p.capacity = 16;
  mr_tree_desc t{};
  t.Jmin = 1; t.Jmax = 1; t.eps = 1e-3; t.ic_kind = MR_IC_GAUSS; t.ic[3] = 0.1;
  mr_ctx c = nullptr;
  if (mr_create(&p, &t, &c) != MR_OK) return 1;
  const int n = 3, T = mr::cnn_tile(17);
  std::vector<float> w(mr::kCnnParams), x(n * 2 * T * T), y(n), prob(n), grad(mr::kCnnParams);
  float loss = 0.f;
  auto eval = [&](int k) {
    calls = queued = 0;
    fail_at = k;
    return mr_cnn_eval(c, w.data(), x.data(), y.data(), n, 1.f, prob.data(), grad.data(), &loss);
  };
  if (eval(0) != MR_OK || queued != 0) return 2;
  const int total = calls;
  for (int k = 1; k <= total; ++k) {
    const int s = eval(k);
    std::printf("%s %d %d\n", name, s, queued);
  }
  std::fflush(stdout);
  std::_Exit(0);
}
