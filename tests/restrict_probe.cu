// A restriction of two right-hand sides at a given width (lanes per row, or 256: a block per row), for
// tests/test_gpu_restrict_widths.py: bc = R x and, with dinv, xc = invtheta dinv bc.  Device arrays; precision 0 FP64, 1 FP32.
#include "../paper_2204_03575_gb300/csrc/amg.cu"

namespace {
template <typename T>
int run(int rows, int cols, const int* rowptr, const int* col, const void* val, const void* x, int width, const void* dinv,
        double invtheta, void* bc, void* xc) {
  using namespace ch;
  using V2 = typename V2T<T>::t;
  Csr<T> R;
  R.nrows = rows;
  R.ncols = cols;
  R.rowptr = const_cast<int*>(rowptr);
  R.col = const_cast<int*>(col);
  R.val = const_cast<T*>(static_cast<const T*>(val));
  launch_restrict_x<T, V2>(width, R, OneVec<V2>{static_cast<const V2*>(x)}, static_cast<V2*>(bc),
                           static_cast<const T*>(dinv), (T)invtheta, static_cast<V2*>(xc), nullptr, false);
  CH_LAUNCHED();
  CH_CUDA(cudaDeviceSynchronize());
  return CH_OK;
}
}  // namespace

extern "C" int restrict_probe(int precision, int rows, int cols, const int* rowptr, const int* col, const void* val,
                              const void* x, int width, const void* dinv, double invtheta, void* bc, void* xc) {
  return precision ? run<float>(rows, cols, rowptr, col, val, x, width, dinv, invtheta, bc, xc)
                   : run<double>(rows, cols, rowptr, col, val, x, width, dinv, invtheta, bc, xc);
}
