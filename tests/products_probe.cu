// The set-up's sparse product and transposition on given matrices (host arrays), for tests/test_gpu_sparse_products.py.
// Return the entry count, negative on an error or where the result has more than `room` entries.
#include "../paper_2204_03575_gb300/csrc/ch_internal.cuh"

namespace {
using namespace ch;
ch_status upload(Alloc& mem, int rows, int cols, const int* rowptr, const int* col, const double* val, Csr<double>* A) {
  A->nrows = rows;
  A->ncols = cols;
  A->nnz = rowptr[rows];
  CH_TRY(mem.get(&A->rowptr, (size_t)rows + 1));
  CH_TRY(mem.get(&A->col, (size_t)A->nnz));
  CH_TRY(mem.get(&A->val, (size_t)A->nnz));
  CH_CUDA(cudaMemcpy(A->rowptr, rowptr, sizeof(int) * (rows + 1), cudaMemcpyHostToDevice));
  CH_CUDA(cudaMemcpy(A->col, col, sizeof(int) * A->nnz, cudaMemcpyHostToDevice));
  CH_CUDA(cudaMemcpy(A->val, val, sizeof(double) * A->nnz, cudaMemcpyHostToDevice));
  return CH_OK;
}
int64_t download(const Csr<double>& C, int64_t room, int* rowptr, int* col, double* val) {
  if (C.nnz > room) return -2;
  if (cudaMemcpy(rowptr, C.rowptr, sizeof(int) * (C.nrows + 1), cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(col, C.col, sizeof(int) * C.nnz, cudaMemcpyDeviceToHost) != cudaSuccess ||
      cudaMemcpy(val, C.val, sizeof(double) * C.nnz, cudaMemcpyDeviceToHost) != cudaSuccess)
    return -3;
  return C.nnz;
}
}  // namespace

extern "C" int64_t product_probe(int n, int k, int m, const int* ap, const int* ac, const double* av, const int* bp,
                                 const int* bc, const double* bv, int64_t room, int* cp, int* cc, double* cv) {
  Alloc mem;
  Csr<double> A, B, C;
  if (upload(mem, n, k, ap, ac, av, &A) != CH_OK || upload(mem, k, m, bp, bc, bv, &B) != CH_OK ||
      spgemm(A, B, &C, nullptr, mem) != CH_OK)
    return -1;
  return download(C, room, cp, cc, cv);
}

extern "C" int64_t transpose_probe(int n, int m, const int* ap, const int* ac, const double* av, int64_t room, int* cp,
                                   int* cc, double* cv) {
  Alloc mem;
  Csr<double> A, C;
  if (upload(mem, n, m, ap, ac, av, &A) != CH_OK || transpose(A, &C, nullptr, mem) != CH_OK) return -1;
  return download(C, room, cp, cc, cv);
}
