// For tests/test_gpu_learned_out_of_memory.py: `steps` learned steps of a state whose allocations are counted, where the
// fail_at-th one of the first such step fails as an exhausted device would (0: none) and that step is called again.
// Returns the failed call's status (0: none failed); the state's N x 4 fields go to x.
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
#include "../paper_2204_03575_gb300/csrc/krylov.cu"

extern "C" int learned_probe(const void* sys, void* pc, void* net, int steps, int fail_at, double* x) {
  using namespace ch;
  ch_state_s* S = nullptr;
  g_left = 0;
  if (state_create(static_cast<const ch_system_s*>(sys), static_cast<ch_precond_s*>(pc), nullptr, &S) != CH_OK ||
      state_seeded(S, 0.33, 0.31, 0.01, 7, nullptr) != CH_OK)
    return -1;
  ch_step_stats stats;
  int failed = 0;
  for (int k = 0; k < steps; ++k) {
    if (k == 0) g_left = fail_at;
    int r = state_step_learned(S, static_cast<ch_ws_s*>(net), nullptr, &stats);
    g_left = 0;
    if (k == 0 && r != CH_OK) {
      failed = r;
      r = state_step_learned(S, static_cast<ch_ws_s*>(net), nullptr, &stats);
    }
    if (r != CH_OK) return -2;
  }
  const bool ok = cudaMemcpy(x, S->x, sizeof(double) * 4 * S->N, cudaMemcpyDeviceToHost) == cudaSuccess;
  state_destroy(S);
  return ok ? failed : -3;
}
