// The two Gram-Schmidt passes and their close on given vectors, for tests/test_gpu_gram_schmidt_close.py: one run of
// N nodes, nv basis vectors V (nv x N x 4), the vector W (N x 4; on return after the first projection), V_{j+1} into
// vnext.  scalars: h1 (2 x 65), h2 (2 x 65), 1 / h_{j+1,j} (2), the column of R (2 x 64, row-major per species).
#include "../paper_2204_03575_gb300/csrc/krylov.cu"

#include <vector>

extern "C" int orth_probe(int N, int nv, int blocks, const double* V, double* W, double* vnext, double* scalars) {
  using namespace ch;
  std::vector<int> run(blocks, 0), lo(blocks), hi(blocks), first = {0, blocks};
  for (int b = 0; b < blocks; ++b) {
    lo[b] = (int)((int64_t)N * b / blocks);
    hi[b] = (int)((int64_t)N * (b + 1) / blocks);
  }
  Alloc mem;
  int *d_run, *d_lo, *d_hi, *d_first;
  unsigned int* tickets;
  double* partials;
  KrylovDev* kd;
  CH_TRY(mem.get(&d_run, blocks));
  CH_TRY(mem.get(&d_lo, blocks));
  CH_TRY(mem.get(&d_hi, blocks));
  CH_TRY(mem.get(&d_first, 2));
  CH_TRY(mem.get(&tickets, blocks));
  CH_TRY(mem.get(&partials, (size_t)2 * blocks * MAXV));
  CH_TRY(mem.get(&kd, 1));
  CH_CUDA(cudaMemcpy(d_run, run.data(), sizeof(int) * blocks, cudaMemcpyHostToDevice));
  CH_CUDA(cudaMemcpy(d_lo, lo.data(), sizeof(int) * blocks, cudaMemcpyHostToDevice));
  CH_CUDA(cudaMemcpy(d_hi, hi.data(), sizeof(int) * blocks, cudaMemcpyHostToDevice));
  CH_CUDA(cudaMemcpy(d_first, first.data(), sizeof(int) * 2, cudaMemcpyHostToDevice));
  CH_CUDA(cudaMemset(tickets, 0, sizeof(unsigned int) * blocks));
  std::vector<KrylovDev> k(1);
  memset(k.data(), 0, sizeof(KrylovDev));
  for (int s = 0; s < 2; ++s) {
    k[0].active[s] = k[0].cycle_active[s] = 1;
    k[0].g[s][nv - 1] = 1.0;
    for (int q = 0; q < nv; ++q) k[0].cs[s][q] = 1.0;  // earlier rotations: none
  }
  CH_CUDA(cudaMemcpy(kd, k.data(), sizeof(KrylovDev), cudaMemcpyHostToDevice));
  const Seg sg{d_run, d_lo, d_hi, d_first, tickets, blocks};
  const double4_32a* V4 = reinterpret_cast<const double4_32a*>(V);
  double4_32a* W4 = reinterpret_cast<double4_32a*>(W);
  k_orth<0><<<blocks, ORTH_TPB>>>(sg, N, nv, V4, W4, partials, kd);
  k_orth<1><<<blocks, ORTH_TPB>>>(sg, N, nv, V4, W4, partials, kd);
  k_orth_close<<<blocks + 1, ORTH_TPB>>>(sg, N, nv, V4, W4, reinterpret_cast<double4_32a*>(vnext), partials,
                                         kd);
  CH_LAUNCHED();
  CH_CUDA(cudaDeviceSynchronize());
  CH_CUDA(cudaMemcpy(k.data(), kd, sizeof(KrylovDev), cudaMemcpyDeviceToHost));
  const size_t nh = 2 * (MAXM + 1);
  memcpy(scalars, k[0].h1, sizeof(double) * nh);
  memcpy(scalars + nh, k[0].h2, sizeof(double) * nh);
  memcpy(scalars + 2 * nh, k[0].hinv, sizeof(double) * 2);
  for (int s = 0; s < 2; ++s)
    for (int q = 0; q < nv; ++q) scalars[2 * nh + 2 + s * MAXM + q] = k[0].R[s][q][nv - 1];
  return 0;
}
