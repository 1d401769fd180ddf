// For tests/test_gpu_train_out_of_memory.py: ws_train_residual on a network whose allocations are counted, with the
// fail_at-th one of the first call failing as an exhausted device would (0: none).  Returns the first call's status; the
// second call, without a failure, gives *loss and the gradients (nparam floats).
#include <cuda_runtime.h>
static int g_left = 0;  // allocations until the failing one
static cudaError_t counted_malloc(void** p, size_t n) {
  if (g_left > 0 && --g_left == 0) {
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  return cudaMalloc(p, n);
}
#define cudaMalloc counted_malloc
#include "../paper_2204_03575_gb300/csrc/warmstart.cu"

extern "C" int train_probe(const void* sys, void* pc, int H, int W, int B, const float* params, const float* norm20,
                           const double* x, const double* q, const double* q2, int fail_at, float* loss, float* grads) {
  using namespace ch;
  ch_ws_s* w = nullptr;
  g_left = 0;
  if (ws_create(H, W, B, &w) != CH_OK || ws_set_params(w, params, nullptr) != CH_OK ||
      ws_set_norm(w, norm20, nullptr) != CH_OK)
    return -1;
  const ch_system_s* s = static_cast<const ch_system_s*>(sys);
  ch_precond_s* p = static_cast<ch_precond_s*>(pc);
  g_left = fail_at;
  const int first = ws_train_residual(w, s, p, x, q, q2, B, 0.f, loss, nullptr);
  g_left = 0;
  *loss = -1.f;
  const int second = ws_train_residual(w, s, p, x, q, q2, B, 0.f, loss, nullptr);
  std::vector<float> host(ws_nparam());
  const int third = ws_get_params(w, host.data(), grads, nullptr);
  ws_destroy(w);
  return second != CH_OK || third != CH_OK ? -2 : first;
}
