// Internal declarations shared by the CUDA translation units of libch.so.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <string>
#include <utility>
#include <vector>

#include "../../include/ch.h"

namespace ch {

// ---------------------------------------------------------------- errors
void set_error(const char* fmt, ...);

#define CH_CUDA(call)                                                                      \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess) {                                                               \
      ::ch::set_error("%s:%d %s: %s", __FILE__, __LINE__, #call, cudaGetErrorString(e_)); \
      return e_ == cudaErrorMemoryAllocation ? CH_ERR_OOM : CH_ERR_CUDA;                   \
    }                                                                                      \
  } while (0)

#define CH_LAUNCHED() CH_CUDA(cudaGetLastError())

#define CH_TRY(call)                \
  do {                              \
    ch_status s_ = (call);          \
    if (s_ != CH_OK) return s_;     \
  } while (0)

#define CH_ARG(cond, msg)                                        \
  do {                                                           \
    if (!(cond)) {                                               \
      ::ch::set_error("invalid argument: %s", msg);              \
      return CH_ERR_ARG;                                         \
    }                                                            \
  } while (0)

// ---------------------------------------------------------------- device memory owned by a handle
struct Alloc {
  std::vector<void*> ptrs;
  Alloc() = default;
  Alloc(const Alloc&) = delete;
  Alloc& operator=(const Alloc&) = delete;
  ~Alloc() { release(); }
  void release() {
    for (void* p : ptrs) cudaFree(p);
    ptrs.clear();
  }
  template <typename T>
  ch_status get(T** out, size_t n) {
    *out = nullptr;
    if (n == 0) n = 1;
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, n * sizeof(T));
    if (e != cudaSuccess) {
      cudaGetLastError();
      set_error("cudaMalloc of %zu bytes failed: %s", n * sizeof(T), cudaGetErrorString(e));
      return e == cudaErrorMemoryAllocation ? CH_ERR_OOM : CH_ERR_CUDA;
    }
    ptrs.push_back(p);
    *out = static_cast<T*>(p);
    return CH_OK;
  }
  void forget(void* p) {  // free one allocation early
    for (size_t i = 0; i < ptrs.size(); ++i)
      if (ptrs[i] == p) {
        cudaFree(p);
        ptrs[i] = ptrs.back();
        ptrs.pop_back();
        return;
      }
  }
};

// ---------------------------------------------------------------- sparse matrices
template <typename T>
struct Csr {
  int nrows = 0, ncols = 0;
  int64_t nnz = 0;
  int* rowptr = nullptr;
  int* col = nullptr;
  T* val = nullptr;
};

constexpr int TPB = 256;  // threads per block of the plain node-parallel kernels
inline int blocks_for(int64_t n, int tpb = TPB) { return (int)((n + tpb - 1) / tpb); }
// fixed grid for deterministic grid-stride reductions: a multiple of the 152 SMs
constexpr int RED_BLOCKS_MAX = 152 * 4;
inline int red_blocks(int64_t n) {
  int b = blocks_for(n);
  return b < RED_BLOCKS_MAX ? (b < 1 ? 1 : b) : RED_BLOCKS_MAX;
}

// ---------------------------------------------------------------- programmatic dependent launch
// A kernel launched with `pdl` set may be scheduled while the kernel before it on the stream is
// still running (its blocks wait in pdl_wait() until that kernel has finished and its writes are
// visible).  The rules every such kernel keeps:
//   - before pdl_wait() it reads only data that no kernel of the current solve writes (operator
//     values, class rows: set-up results) and writes no global memory;
//   - it calls pdl_trigger(), which lets its own successor be scheduled, only after pdl_wait(), so
//     that when the successor's blocks start every kernel but this one has finished.  Without the
//     call the successor is scheduled when this kernel's blocks have all exited (still before
//     the memory flush that pdl_wait() covers).
// Launched without the attribute (pdl = 0, per-launch timing with events between kernels) both
// instructions return at once and the kernel behaves as a plain launch.  No arithmetic changes.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

bool prof_timing();  // prof.cu: per-launch event timing on (launches then stay plain)
template <typename... KArgs, typename... Args>
inline void launch_k(bool pdl, void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     Args&&... args) {
  if (!pdl || prof_timing()) {
    k<<<grid, block, smem, st>>>(std::forward<Args>(args)...);
    return;
  }
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);  // errors reach cudaGetLastError
}

// ---------------------------------------------------------------- primitives (sparse.cu)
// rowptr (n + 1) = exclusive scan of the counts; returns the total in *total (host)
ch_status scan_i32_to_rowptr(const int* counts, int* rowptr, int n, int64_t* total,
                             cudaStream_t st, Alloc& tmp);
// incidence lists: for each of nitems items with k entries (ids in [0,nkeys)), build the
// key -> sorted item list (CSR)
ch_status build_incidence(const int* items, int nitems, int k, int nkeys, int** ptr, int** list,
                          cudaStream_t st, Alloc& mem);
// C = A * B (fp64, deterministic), allocated in mem
ch_status spgemm(const Csr<double>& A, const Csr<double>& B, Csr<double>* C, cudaStream_t st,
                 Alloc& mem);
// B = A^T (fp64), allocated in mem
ch_status transpose(const Csr<double>& A, Csr<double>* B, cudaStream_t st, Alloc& mem);

// ---------------------------------------------------------------- launch accounting (prof.cu)
enum KernelId {
  K_RHS, K_LOADS, K_APPLY_A, K_RESIDUAL4, K_ORTH0, K_ORTH1, K_ORTH2, K_SCALE4, K_UPDATE_X,
  K_CYCLE_SOLVE, K_FLAGS, K_MASS, K_CHEB_FIRST, K_CHEB_STEP, K_VRESIDUAL, K_RESTRICT, K_PROLONG,
  K_COARSE, K_VLOAD, K_VSTORE, K_SPMV_M, K_STATE_IO,
  // the same V-cycle kernels on levels below the finest (accounted separately)
  K_CHEB_FIRST_C, K_CHEB_STEP_C, K_VRESIDUAL_C, K_RESTRICT_C, K_PROLONG_C,
  K_WS_CONV, K_WS_IO, K_GUESS, K_ELEM_LOADS, K_MR_DOT, K_MR_VEC, K_CHEB_SEMI, K_MORPH, K_ORTH_RE, K_COUNT
};
// RAII around one kernel launch: counts it with its algorithmic bytes / FMAs and, when timing
// is on, records CUDA events around it on the launching stream.
class ProfScope {
 public:
  ProfScope(cudaStream_t st, int kid, int f32, double bytes, double fmas);
  ~ProfScope();
  ProfScope(const ProfScope&) = delete;
  ProfScope& operator=(const ProfScope&) = delete;

 private:
  cudaStream_t st_;
  int slot_;
  double bytes_, fmas_;
  cudaEvent_t e0_ = nullptr, e1_ = nullptr;
};
void prof_drain();
bool prof_timing();
// launch accounting of kernels recorded into a CUDA graph, replayed at each graph launch
struct ProfTally {
  int64_t launches[K_COUNT * 2] = {};
  double bytes[K_COUNT * 2] = {};
  double fmas[K_COUNT * 2] = {};
};
// the tally that ProfScopes record into while capturing (nullptr: none); returns the previous one
ProfTally* prof_capture_swap(ProfTally* t);
void prof_add(const ProfTally& t);
void prof_add_times(const ProfTally& t, int64_t times);
// add to one kernel's counters directly (work whose size only the device knew)
void prof_add_slot(int kid, int f32, int64_t launches, double bytes, double fmas);

}  // namespace ch

// ---------------------------------------------------------------- lattice classes of a uniform mesh
namespace ch {
// On a box mesh an assembled row depends only on the widths of the cells on either side of the node along
// each axis (none beyond a rim).  Every node carries a class id and a fine-level operator is one table row
// per id instead of one value per stored entry.  Two partitions of a run's nodes:
//   ch_mesh_s::lat  by the pairs of widths as the node coordinates have them.  Coordinates are rounded, so
//                   the widths of a uniform axis take two values per binade: 3 pairs for 512 cells of 1 / 512,
//                   24 for 799 cells on [0, 10].  The rows of a class are equal bit for bit.
//   ch_mesh_s::pos  by position alone: the first, an inner or the last node along each axis, 9 classes in 2D
//                   and 27 in 3D.  The rows of a class agree to the rounding of the coordinates (1e-13 of an
//                   entry for those 799 cells): below FP32's rounding, and used by FP32 V-cycles only.
struct Lattice {
  int dim = 0;
  int ncls = 0;                 // pos: 9 (2D) or 27 (3D) classes per run
  int nids = 0;                 // classes of all runs
  int multi = 0;                // several runs: the strides are the id's
  int W = 0, WH = 0;            // strides nx + 1 and (nx + 1)(ny + 1) of a single run
  int id32 = 0;                 // ids are 32-bit (more than 65536 of them), else 16-bit
  void* id = nullptr;           // N class ids
  int2* wh = nullptr;           // nids: strides of the id's run
  int* rep = nullptr;           // nids: a node of the class
};
// The grid of one run: first node, first cell, cells per axis.
struct CellGrid {
  int node0, cell0, nx, ny, nz;
};
// strides of the lattice directions: 7 in 2D (the triangles' edges), 15 in 3D (the Kuhn tetrahedra's),
// ascending for any W, H >= 2, i.e. in CSR column order; direction ND / 2 is the node itself
__host__ __device__ __forceinline__ int lat_off(int nd, int d, int W, int WH) {
  constexpr int a2[7] = {-1, 0, -1, 0, 1, 0, 1}, b2[7] = {-1, -1, 0, 0, 0, 1, 1};
  constexpr int a3[15] = {-1, 0, -1, 0, -1, 0, -1, 0, 1, 0, 1, 0, 1, 0, 1};
  constexpr int b3[15] = {-1, -1, 0, 0, -1, -1, 0, 0, 0, 1, 1, 0, 0, 1, 1};
  constexpr int c3[15] = {-1, -1, -1, -1, 0, 0, 0, 0, 0, 0, 0, 1, 1, 1, 1};
  return nd == 7 ? a2[d] + b2[d] * W : a3[d] + b3[d] * W + c3[d] * WH;
}
__device__ __forceinline__ int lat_id(const Lattice& L, int i) {
  return L.id32 ? static_cast<const int*>(L.id)[i] : static_cast<const uint16_t*>(L.id)[i];
}

// The block operator of Eq. (14) on the lattice: per class id a table row of the mass entries m_d and of
// the stiffness entries k_e over the axis directions e -- the only ones where the stiffness matrix of a box
// mesh is not zero (5 of 7 in 2D, 7 of 15 in 3D).  The entries are the assembled ones (set-up check, bit
// for bit); tab is null where they are not, and the CSR form is taken: entries below FP64's normal range.
struct LatOperator {
  Lattice L;
  double a = 0, c = 0;
  const double* tab = nullptr;
};
template <int ND> struct LatAxes;
template <> struct LatAxes<7> {
  static constexpr int NK = 5, TS = 12;  // axis directions; doubles per table row (ND + NK, even)
  __host__ __device__ static constexpr int index(int d) { return d >= 1 && d <= 5 ? d - 1 : -1; }
};
template <> struct LatAxes<15> {
  static constexpr int NK = 7, TS = 22;
  __host__ __device__ static constexpr int index(int d) {
    constexpr int k[15] = {-1, -1, -1, 0, -1, 1, 2, 3, 4, 5, -1, 6, -1, -1, -1};
    return k[d];
  }
};

// (A x)_i for both species: y1 = M x1 + a K x2, y2 = a K x1 - c M x2, in the order and with the roundings of
// the CSR form (products m c and k a formed beforehand, six instructions fewer, rounded 1.2 to 1.5 times as
// far from the exact sum).  4 FMAs per direction, 4 more per axis direction and 6 at the end (54 in 2D, 94 in
// 3D, against 8 per stored entry, 62 and 126, in CSR form).
template <int ND>
__device__ __forceinline__ double4_32a lat_apply_A(const LatOperator& A, int i, const double4_32a* __restrict__ x) {
  using X = LatAxes<ND>;
  const int id = lat_id(A.L, i);
  int W = A.L.W, WH = A.L.WH;
  if (A.L.multi) {
    const int2 w = A.L.wh[id];
    W = w.x;
    WH = w.y;
  }
  const double2* row = reinterpret_cast<const double2*>(A.tab + (size_t)id * X::TS);
  double t[X::TS];
#pragma unroll
  for (int q = 0; q < X::TS / 2; ++q) {
    const double2 v = row[q];
    t[2 * q] = v.x;
    t[2 * q + 1] = v.y;
  }
  double4_32a m = make_double4_32a(0.0, 0.0, 0.0, 0.0), k = m;
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    // a neighbour the class lacks (mass entry zero) is not read: it would be another row's or run's value
    double4_32a z = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    if (__double2hiint(t[d]) != 0) z = x[i + lat_off(ND, d, W, WH)];
    m.x = fma(t[d], z.x, m.x);
    m.y = fma(t[d], z.y, m.y);
    m.z = fma(t[d], z.z, m.z);
    m.w = fma(t[d], z.w, m.w);
    if (X::index(d) >= 0) {
      const double s = t[ND + (X::index(d) >= 0 ? X::index(d) : 0)];
      k.x = fma(s, z.x, k.x);
      k.y = fma(s, z.y, k.y);
      k.z = fma(s, z.z, k.z);
      k.w = fma(s, z.w, k.w);
    }
  }
  return make_double4_32a(fma(A.a, k.z, m.x), fma(A.a, k.w, m.y), fma(A.a, k.x, -A.c * m.z),
                          fma(A.a, k.y, -A.c * m.w));
}
}  // namespace ch

// ---------------------------------------------------------------- opaque handles
struct ch_mesh_s {
  ch_params p{};                 // parameters of run 0 (the only run of a plain mesh)
  std::vector<ch_params> runs;   // per-run parameters (box, cells)
  bool batch = false;            // built by ch_mesh_batch
  std::vector<int> run_off;      // host: first node of each run, run_off[R] = N
  int* run_off_d = nullptr;      // device copy
  int* node_run = nullptr;       // run of each node
  int dim = 2, N = 0, E = 0, Fb = 0, Ft = 0;
  double* coords = nullptr;   // N x dim
  int* elems = nullptr;       // E x (dim+1)
  int* bot = nullptr;         // Fb x dim
  int* top = nullptr;         // Ft x dim
  double* vol = nullptr;      // E element measures
  double* bvol = nullptr;     // Fb facet measures
  double* tvol = nullptr;     // Ft facet measures
  int *n2e_ptr = nullptr, *n2e = nullptr;  // node -> incident elements (sorted)
  int *n2b_ptr = nullptr, *n2b = nullptr;  // node -> incident bottom facets
  int *n2t_ptr = nullptr, *n2t = nullptr;  // node -> incident top facets
  ch::Lattice lat, pos;  // classes by cell widths, by position
  ch::CellGrid* cell_grid = nullptr;  // device, per run
  ch::Alloc mem;
};

struct ch_system_s {
  const ch_mesh_s* mesh = nullptr;
  ch_params p{};
  int N = 0;
  int64_t nnz = 0;
  int* rowptr = nullptr;
  int* col = nullptr;
  double* valM = nullptr;
  double* valK = nullptr;
  double* valH = nullptr;
  int* diag = nullptr;  // position of the diagonal entry of each row
  double2* eload = nullptr;  // per grid cell and corner, the f-load contributions (polymer, NFA)
  void* log_tables = nullptr;  // potential = 3: the load's logarithm tables
  double* bw = nullptr;     // pattern = 1: Fb x 2 species x (dim + dim^2) substrate weights, else null
  double a = 0, c = 0;  // A = [[M, aK], [aK, -cM]]
  ch::LatOperator lat;  // ... on the lattice
  ch::Alloc mem;
};

namespace ch {
struct Hierarchy;  // amg.cu
ch_status hierarchy_build(const Csr<double>& A0, const ch_mesh_s* mesh, const ch_params& p, int precision,
                          cudaStream_t st, Hierarchy** out);
void hierarchy_free(Hierarchy* h);
int hierarchy_levels(const Hierarchy* h);
void hierarchy_level_size(const Hierarchy* h, int l, int64_t* rows, int64_t* nnz);
ch_status hierarchy_level_export(const Hierarchy* h, int l, int64_t* rows, int64_t* nnz, int64_t* nnz_P,
                                 double* lo, double* hi, int* degree, int* A_rowptr, int* A_col,
                                 double* A_val, int* P_rowptr, int* P_col, double* P_val, cudaStream_t st);
void hierarchy_level_tiles(const Hierarchy* h, int l, int* tA, int* tR, int* tP);
// x (N x 2, fp64, row stride ldx) ~ A^-1 b (N x 2, fp64, row stride ldb), ncyc V-cycles
ch_status hierarchy_solve(Hierarchy* h, const double* b, int ldb, double* x, int ldx, int ncyc,
                          cudaStream_t st);
// x (N x 2, fp64, read and overwritten) after `passes` passes of the finest level's Chebyshev smoother
ch_status hierarchy_smooth(Hierarchy* h, const double* b, double* x, int degree, int passes, cudaStream_t st);
// as hierarchy_solve (strides 2), work vectors in a static device array: no device allocation
ch_status hierarchy_solve_noalloc(Hierarchy* h, const double* b, double* x, int ncyc, cudaStream_t st);

// assemble.cu
ch_status loads(const ch_system_s* s, const double* pp, const double* pn, double* Fp, double* Fn,
                double* gp, double* gn, cudaStream_t st);
// b (N x 4) from phi_p, phi_nfa read with element stride ld
ch_status rhs_strided(const ch_system_s* s, const double* pp, const double* pn, int ld, double* b,
                      cudaStream_t st);
ch_status mesh_build(ch_mesh_s* m, cudaStream_t st);
ch_status assemble_system(const ch_mesh_s* m, ch_system_s* s, cudaStream_t st);
ch_status apply_A(const ch_system_s* s, const double* x, double* y, cudaStream_t st);
}  // namespace ch

struct ch_precond_s {
  const ch_system_s* sys = nullptr;
  int precision = 0;
  ch::Hierarchy* hM = nullptr;
  ch::Hierarchy* hH = nullptr;
  double* t1 = nullptr;  // N x 2 temporaries for Algorithm 1
  double* t2 = nullptr;
  cudaStream_t side = nullptr;  // Algorithm 1's M-solve branch (non-blocking)
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  ch::Alloc mem;
  ~ch_precond_s() {
    ch::hierarchy_free(hM);
    ch::hierarchy_free(hH);
    if (ev_fork) cudaEventDestroy(ev_fork);
    if (ev_join) cudaEventDestroy(ev_join);
    if (side) cudaStreamDestroy(side);
  }
};

struct ch_state_s;
namespace ch {
ch_status precond_apply(ch_precond_s* pc, const double* v, double* w, cudaStream_t st);
// Algorithm 1's step 1 on two right-hand sides (N x 2 fp64): x = M~^-1 b
ch_status mass_solve(ch_precond_s* pc, const double* b, double* x, cudaStream_t st);
// morphology.cu: Section 5's projection of a thresholded 2D morphology onto a finite-difference grid
ch_status morphology_project(const double* pp, const double* pn, int nx, int ny, double Lx, double Ly,
                             int use_thr, double thr, int gx, int gy, uint8_t* polymer, double* mu_e,
                             double* mu_h, cudaStream_t st);
const char* last_error();
ch_status state_create(const ch_system_s* s, ch_precond_s* pc, cudaStream_t st, ch_state_s** out);
void state_destroy(ch_state_s* S);
ch_status state_set(ch_state_s* S, const double* pp, const double* pn, const double* mp,
                    const double* mn, cudaStream_t st);
ch_status state_seeded(ch_state_s* S, double p0, double n0, double noise, uint64_t seed,
                       cudaStream_t st);
ch_status state_get(const ch_state_s* S, double* pp, double* pn, double* ps, double* mp, double* mn,
                    cudaStream_t st);
ch_status state_seeded_batch(ch_state_s* S, const double* base_p, const double* base_n, double noise,
                             uint64_t seed, cudaStream_t st);
ch_status state_run_stats(const ch_state_s* S, int run, ch_step_stats* out);
ch_status state_save(const ch_state_s* S, const char* path, cudaStream_t st);
ch_status state_load(ch_state_s* S, const char* path, cudaStream_t st);
ch_status state_step(ch_state_s* S, cudaStream_t st, ch_step_stats* stats);
}

// warmstart.cu
struct ch_ws_s;
namespace ch {
ch_status ws_create(int H, int W, int Bmax, ch_ws_s** out);
// convolution engine: 0 mma.sync, 1 tcgen05; ws_check reports a timed-out tcgen05 block (call
// after synchronising with the network's work)
ch_status ws_set_engine(ch_ws_s* w, int engine);
ch_status ws_withhold_mma(ch_ws_s* w, int on);
ch_status ws_check(const ch_ws_s* w);
void ws_destroy(ch_ws_s* w);
ch_status ws_set_params(ch_ws_s* w, const float* host, cudaStream_t st);
ch_status ws_get_params(const ch_ws_s* w, float* host, float* host_grads, cudaStream_t st);
ch_status ws_set_norm(ch_ws_s* w, const float* host20, cudaStream_t st);
ch_status ws_fit_norm(ch_ws_s* w, const void* x, int S, int fp32, double* host20, cudaStream_t st);
ch_status ws_predict(ch_ws_s* w, const double* state, const double* prev, const double* prev2, double* pred,
                     cudaStream_t st);
ch_status ws_train_step(ch_ws_s* w, const float* x, const float* q, const float* q2, const float* n, int B,
                        float lap, float lr, float* loss, cudaStream_t st);
ch_status ws_train_residual(ch_ws_s* w, const ch_system_s* sys, ch_precond_s* pc, const double* x,
                            const double* q, const double* q2, int B, float lr, float* loss, cudaStream_t st);
int ws_nparam();
void ws_dims(const ch_ws_s* w, int* H, int* W);
ch_status state_step_learned(ch_state_s* S, ch_ws_s* w, cudaStream_t st, ch_step_stats* stats);
ch_status state_step_guess(ch_state_s* S, const double* guess, cudaStream_t st, ch_step_stats* stats);
}  // namespace ch
