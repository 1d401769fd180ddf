// Algebraic multigrid for the inner solves of Algorithm 1 (M~ ~ M and H = aK + sqrt(c)M).
//
// The paper uses Ruge-Stueben AMG from a CPU library (Section 4).  Here the hierarchy is
// built on the device by smoothed aggregation (Vanek, Mandel, Brezina 1996) with MIS(2)
// aggregates found by the parallel maximal-independent-set method of Bell, Dalton and
// Olson (2012):
//   strength  |a_ij| >= theta sqrt(a_ii a_jj), plus each row's strongest entry, symmetrised;
//   MIS(2)    random-priority independent set at graph distance 2, roots become aggregates;
//   P         (I - omega D^-1 A) T with T the aggregate indicator, omega = 4/(3 rho),
//             rho = min(Gershgorin bound, 1.05 x power-iteration estimate) of lambda_max(D^-1 A);
//   A_c       = P^T A P (deterministic sparse products), down to <= coarse_max rows, whose
//             dense inverse is formed on the device.
// Smoothing is Chebyshev on D^-1 A over [cheb_lower, 1] * 1.1 rho, with the same rho.  Every set-up sum has a fixed
// order, so the hierarchy is bitwise reproducible.  V-cycles run in FP64 or FP32 on two
// right-hand sides at once (the two species share M and H).
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <set>
#include <tuple>
#include <type_traits>

#include "ch_internal.cuh"

namespace ch {

template <typename T> struct V2T;
template <> struct V2T<double> { using t = double2; };
template <> struct V2T<float> { using t = float2; };

// Fine-level operator of a uniform mesh in lattice form: node i's neighbours sit at i + lat_off(d)
// and its row is the table row of its class id (Lattice): nd values in ascending direction, i.e. in
// CSR column order (zero where the class has no such neighbour: the clamped index is then read but
// multiplied by zero), padded to `ts` with the class's factor in slot nd.  FP64 V-cycles take the classes
// by cell widths, whose rows are the assembled ones bit for bit; FP32 V-cycles the few classes by position
// where the rows of a class agree to 2^-36 of the diagonal, far below FP32's rounding (checked at set-up),
// or else those by widths.
template <typename T>
struct LatOp {
  int nd = 0;                      // 7 (2D) or 15 (3D); 0: not structured, use the CSR form
  int ts = 0;                      // values per table row: 8 or 16
  Lattice L;
  const T* tab = nullptr;          // nids x ts: the operator's rows (slot nd: 1 / diagonal)
};

// One tile of the 2D lattice form for k_smooth_tile: the run's first node, strides and ids, and the
// tile's first output column and row.
struct LatTile {
  int off, W, H, x0, y0, id0;
};
// columns of a region, nodes per thread, groups (thread rows) of a block at most, and of a block that
// shares its SM with another
template <typename T> struct TileShape;
template <> struct TileShape<float> { static constexpr int RW = 64, ROWS = 4, GMAX = 12, GPAIR = 8; };
template <> struct TileShape<double> { static constexpr int RW = 16, ROWS = 1, GMAX = 16, GPAIR = 16; };
// FP64 passes are bound by the FP64 pipe, where recomputed halo nodes cost as much as any: tiles only
// while the mesh gives the chip at most two per SM and a step is a launch's latency (us per application
// of Algorithm 1 with tiles / a launch per step: 32 x 32 90 / 146, 64 x 64 164 / 214; 96 x 96 with four
// tiles per SM took a third more than by steps)
constexpr int TILE_MAX_F64 = 304;
struct TilePlan {
  int ntiles = 0;     // 0: the pass runs as one launch per step
  int groups = 0;     // thread rows of a block
  int halo = 0;       // operator applications of the pass
  bool pair = false;  // two blocks share an SM
  const LatTile* tiles = nullptr;
};

template <typename T>
struct LevelT {
  Csr<T> A, P, R;
  Csr<T> RB;  // [R, -R A] over the stacked (b, x): the coarse right-hand side without the residual
  LatOp<T> lat;                        // level 0 of a box mesh
  TilePlan plan, plan_r;               // ... its smoothing passes as single launches, and those from a
                                       // given iterate that also form the residual
  int tprA = 1, tprP = 1, tprR = 1;  // lanes per row of the SpMV-type kernels (autotuned)
  bool pdl = false;                  // launch the V-cycle kernels as programmatic dependents
  T* dinv = nullptr;
  typename V2T<T>::t *x = nullptr, *x2 = nullptr, *r = nullptr, *b = nullptr;
};

struct Hierarchy {
  int precision = 0;
  int nlev = 0;
  std::vector<Csr<double>> A, P, R;  // FP64 set-up results
  std::vector<Csr<double>> RA;       // R A where the cycle restricts with it (set-up only)
  std::vector<double*> dinv;
  std::vector<double> rho;            // per level: min(Gershgorin bound, 1.05 x power estimate) of
                                      // lambda_max(D^-1 A); Chebyshev interval [lower, 1] x 1.1 rho
  std::vector<LevelT<double>> Ld;     // working copies (precision 0)
  std::vector<LevelT<float>> Lf;      // working copies (precision 1)
  int nc = 0;                         // coarsest size
  double* cinv = nullptr;             // nc x nc dense inverse (FP64)
  float* cinvf = nullptr;
  int cheb_degree = 2;
  int cheb_degree_coarse = 2;         // on the levels below the finest
  double cheb_lower = 0.3;
  int autotune = 1;
  bool pdl = true;
  Alloc mem;
};

// ---------------------------------------------------------------- set-up kernels
__global__ void k_diag_gersh(Csr<double> A, double* dinv, double* rowbound) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  double d = 0.0, s = 0.0;
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) {
    if (A.col[q] == i) d = A.val[q];
    s += fabs(A.val[q]);
  }
  dinv[i] = 1.0 / d;
  rowbound[i] = s / fabs(d);
}

// *out (0 on entry) = max over v of non-negative values: their bit patterns order like integers
__global__ void k_max_reduce(const double* v, int n, unsigned long long* out) {
  double m = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) m = fmax(m, v[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0 && m > 0.0) atomicMax(out, (unsigned long long)__double_as_longlong(m));
}

__global__ void k_abs_diag(int n, const double* dinv, double* d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = fabs(1.0 / dinv[i]);
}

// nrm: nnz scratch (each entry's normalised size is formed once: an FP64 square root and division)
__global__ void k_strength(Csr<double> A, const double* dabs, double theta, double* nrm, uint8_t* s) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  const double di = dabs[i];
  double mx = 0.0;
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) {
    const int j = A.col[q];
    if (j == i) continue;
    const double v = fabs(A.val[q]) / sqrt(di * dabs[j]);
    nrm[q] = v;
    mx = fmax(mx, v);
  }
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) {
    uint8_t st = 0;
    if (A.col[q] != i) {
      const double v = nrm[q];
      st = (v >= theta || (mx > 0.0 && v >= mx)) ? 1 : 0;
    }
    s[q] = st;
  }
}

__device__ __forceinline__ int find_in_row(const int* col, int b, int e, int c) {
  while (b < e) {
    const int m = (b + e) >> 1;
    if (col[m] < c) b = m + 1;
    else e = m;
  }
  return b;
}

// s2_ij = s_ij or s_ji (A has a symmetric pattern)
__global__ void k_strength_sym(Csr<double> A, const uint8_t* s, uint8_t* s2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) {
    const int j = A.col[q];
    uint8_t v = s[q];
    if (!v && j != i) {
      const int p = find_in_row(A.col, A.rowptr[j], A.rowptr[j + 1], i);
      if (p < A.rowptr[j + 1] && A.col[p] == i) v = s[p];
    }
    s2[q] = v;
  }
}

__device__ __forceinline__ uint32_t hash32(uint32_t x) {  // integer hash (avalanche mixer)
  x ^= x >> 16;
  x *= 0x7feb352dU;
  x ^= x >> 15;
  x *= 0x846ca68bU;
  x ^= x >> 16;
  return x;
}

// key = state (2 bits) | hash (32 bits) | index (30 bits); state 2 = in, 1 = undecided, 0 = out
__device__ __forceinline__ uint64_t mis_key(int state, int i) {
  return ((uint64_t)state << 62) | ((uint64_t)hash32((uint32_t)i) << 30) | (uint64_t)i;
}

__global__ void k_mis_keys(int n, const int8_t* state, uint64_t* key) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) key[i] = mis_key(state[i], i);
}

__global__ void k_strong_max(Csr<double> A, const uint8_t* s, const uint64_t* in, uint64_t* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  uint64_t m = in[i];
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q)
    if (s[q]) {
      const uint64_t v = in[A.col[q]];
      m = v > m ? v : m;
    }
  out[i] = m;
}

__global__ void k_mis_update(int n, const uint64_t* key, const uint64_t* m2, int8_t* state,
                             int* undecided) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || state[i] != 1) return;
  if (m2[i] == key[i]) state[i] = 2;
  else if ((m2[i] >> 62) == 2) state[i] = 0;
  else atomicAdd(undecided, 1);
}

__global__ void k_roots(int n, const int8_t* state, int* isroot) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) isroot[i] = state[i] == 2 ? 1 : 0;
}

// pass 1: roots own aggregate id (scan of isroot); other nodes join the strongest-key
// neighbouring root.  pass >= 2: unassigned nodes join the aggregate of the max-key
// assigned neighbour (reading the previous pass only).
__global__ void k_agg_pass(Csr<double> A, const uint8_t* s, const int* isroot, const int* rootid,
                           const int* agg_in, int* agg_out, int first, int* unassigned) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  if (first) {
    if (isroot[i]) {
      agg_out[i] = rootid[i];
      return;
    }
  } else if (agg_in[i] >= 0) {
    agg_out[i] = agg_in[i];
    return;
  }
  uint64_t best = 0;
  int bj = -1;
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) {
    if (!s[q]) continue;
    const int j = A.col[q];
    const bool ok = first ? (isroot[j] != 0) : (agg_in[j] >= 0);
    if (!ok) continue;
    const uint64_t k = mis_key(0, j);
    if (bj < 0 || k > best) {
      best = k;
      bj = j;
    }
  }
  if (bj >= 0) agg_out[i] = first ? rootid[bj] : agg_in[bj];
  else {
    agg_out[i] = -1;
    atomicAdd(unassigned, 1);
  }
}

// P row i = sum_j (delta_ij - omega a_ij / a_ii) e_{agg(j)}: sort (agg, coef) pairs of row i
// by aggregate (stable insertion sort in a scratch laid out like A) and merge duplicates.
template <bool FILL>
__global__ void k_prolong(Csr<double> A, const double* dinv, const int* agg, double omega,
                          int* skey, double* sval, int* cnt, const int* pptr, int* pcol,
                          double* pval) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  const int b = A.rowptr[i], e = A.rowptr[i + 1];
  for (int q = b; q < e; ++q) {
    const int j = A.col[q];
    const int k = agg[j];
    const double c = (j == i ? 1.0 : 0.0) - omega * A.val[q] * dinv[i];
    int t = q - 1;
    while (t >= b && skey[t] > k) {
      skey[t + 1] = skey[t];
      sval[t + 1] = sval[t];
      --t;
    }
    skey[t + 1] = k;
    sval[t + 1] = c;
  }
  int out = FILL ? pptr[i] : 0, n = 0;
  for (int q = b; q < e; ++q) {
    if (q == b || skey[q] != skey[q - 1]) {
      if (FILL) {
        pcol[out + n] = skey[q];
        pval[out + n] = sval[q];
      }
      ++n;
    } else if (FILL) {
      pval[out + n - 1] += sval[q];
    }
  }
  if (!FILL) cnt[i] = n;
}

// D (n x n, zeroed) = A
__global__ void k_to_dense(Csr<double> A, double* D) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) D[(size_t)i * A.nrows + A.col[q]] = A.val[q];
}

// In-place inverse of the SPD n x n matrix D by block Gauss-Jordan elimination, GJ_B pivots at a time
// (no pivoting needed; a non-positive pivot is reported).  With K the block's rows and columns, L =
// D[:, K] and P = D[K, K]^-1:
//   k_gj_panel:  R = P D[K, :] with R[:, K] = P, and a copy of L (the update overwrites it),
//   k_gj_update: D[i, :] = (D[i, :] with columns K zeroed) - L[i] R for rows outside K, D[K, :] = R.
// Two launches per block instead of two per pivot, n^3 FMAs instead of 2 n^3 on [D | I].  Measured on
// the two coarsest levels of a 256 x 256 set-up (296 and 250 rows or so): 0.69 ms, against 2.35 ms one
// pivot at a time.
constexpr int GJ_B = 32;
__global__ void __launch_bounds__(256) k_gj_panel(int n, int k0, const double* __restrict__ D, double* __restrict__ R,
                                                  double* __restrict__ L, int* bad) {
  __shared__ double P[GJ_B][GJ_B + 1], col[GJ_B], T[GJ_B][GJ_B + 1];
  const int nb = min(GJ_B, n - k0), tid = threadIdx.x;
  for (int e = tid; e < GJ_B * GJ_B; e += 256) {
    const int i = e / GJ_B, j = e % GJ_B;
    P[i][j] = (i < nb && j < nb) ? D[(size_t)(k0 + i) * n + k0 + j] : (i == j ? 1.0 : 0.0);
  }
  __syncthreads();
  for (int k = 0; k < nb; ++k) {  // every block inverts the diagonal block for itself
    const double piv = P[k][k];
    if (tid < GJ_B) col[tid] = P[tid][k];
    if (tid == 0 && blockIdx.x == 0 && !(piv > 0.0)) *bad = 1;
    __syncthreads();
    const double ip = 1.0 / piv;
    if (tid < GJ_B) P[k][tid] = tid == k ? ip : P[k][tid] * ip;
    __syncthreads();
    for (int e = tid; e < GJ_B * GJ_B; e += 256) {
      const int i = e / GJ_B, j = e % GJ_B;
      if (i != k) P[i][j] = (j == k ? 0.0 : P[i][j]) - col[i] * P[k][j];
    }
    __syncthreads();
  }
  // this block's 32 columns of R and 32 rows of L
  const int c0 = blockIdx.x * GJ_B;
  for (int e = tid; e < GJ_B * GJ_B; e += 256) {
    const int i = e / GJ_B, j = e % GJ_B;
    T[i][j] = (i < nb && c0 + j < n) ? D[(size_t)(k0 + i) * n + c0 + j] : 0.0;
    if (c0 + i < n) L[(size_t)(c0 + i) * GJ_B + j] = j < nb ? D[(size_t)(c0 + i) * n + k0 + j] : 0.0;
  }
  __syncthreads();
  for (int e = tid; e < GJ_B * GJ_B; e += 256) {
    const int i = e / GJ_B, j = e % GJ_B, c = c0 + j;
    if (c >= n) continue;
    double r;
    if (c >= k0 && c < k0 + nb) {
      r = P[i][c - k0];
    } else {
      r = 0.0;
      for (int k = 0; k < nb; ++k) r = fma(P[i][k], T[k][j], r);
    }
    R[(size_t)i * n + c] = i < nb ? r : 0.0;
  }
}

// one 32 x 32 tile of D per block (blockIdx.x: columns, blockIdx.y: rows)
__global__ void __launch_bounds__(256) k_gj_update(int n, int k0, double* __restrict__ D, const double* __restrict__ R,
                                                   const double* __restrict__ L) {
  __shared__ double Ls[GJ_B][GJ_B + 1], Rs[GJ_B][GJ_B + 1];
  const int nb = min(GJ_B, n - k0), tid = threadIdx.x;
  const int i0 = blockIdx.y * GJ_B, c0 = blockIdx.x * GJ_B;
  for (int e = tid; e < GJ_B * GJ_B; e += 256) {
    const int i = e / GJ_B, j = e % GJ_B;
    Ls[i][j] = i0 + i < n ? L[(size_t)(i0 + i) * GJ_B + j] : 0.0;
    Rs[i][j] = c0 + j < n ? R[(size_t)i * n + c0 + j] : 0.0;
  }
  __syncthreads();
  for (int e = tid; e < GJ_B * GJ_B; e += 256) {
    const int i = e / GJ_B, j = e % GJ_B, r = i0 + i, c = c0 + j;
    if (r >= n || c >= n) continue;
    double* d = D + (size_t)r * n + c;
    if (r >= k0 && r < k0 + nb) {
      *d = R[(size_t)(r - k0) * n + c];
    } else {
      double t = 0.0;
#pragma unroll 8
      for (int k = 0; k < GJ_B; ++k) t = fma(Ls[i][k], Rs[k][j], t);
      *d = ((c >= k0 && c < k0 + nb) ? 0.0 : *d) - t;
    }
  }
}

__global__ void k_d2f(const double* a, float* b, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (float)a[i];
}
template <typename T>
__global__ void k_copy_cast(const double* a, T* b, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (T)a[i];
}

// B = [R, -RA], a warp per row
template <typename T>
__global__ void k_stack(Csr<double> R, Csr<double> RA, Csr<T> B) {
  const int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32, lane = threadIdx.x & 31;
  if (i >= R.nrows) return;
  const int r0 = R.rowptr[i], r1 = R.rowptr[i + 1], q0 = RA.rowptr[i], q1 = RA.rowptr[i + 1];
  if (lane == 0) B.rowptr[i] = r0 + q0;
  if (lane == 1 && i == R.nrows - 1) B.rowptr[i + 1] = r1 + q1;
  const int o = r0 + q0, o2 = r1 + q0;
  for (int k = r0 + lane; k < r1; k += 32) {
    B.col[o + k - r0] = R.col[k];
    B.val[o + k - r0] = (T)R.val[k];
  }
  for (int k = q0 + lane; k < q1; k += 32) {
    B.col[o2 + k - q0] = R.ncols + RA.col[k];
    B.val[o2 + k - q0] = (T)-RA.val[k];
  }
}

// ---------------------------------------------------------------- spectral radius of D^-1 A
// Power iteration with the D-weighted Rayleigh quotient lambda = (x, A x) / (x, D x), which for
// symmetric A converges twice as fast as the norm ratio.  One launch per iteration: y = D^-1 A x with x
// the previous y times its scale, the block partials of (x, A x), (x, D x) and (y, D y), and in the last
// block their sums (a fixed order), which give lambda and y's scale to D-norm 1.
constexpr int POW_BLOCKS = 152 * 2;

__global__ void k_pow_init(int n, double* x, double* out, unsigned int* ticket) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = 0.5 + (double)(hash32((uint32_t)i * 2654435761u + 12345u) >> 8) * 0x1.0p-24;
  if (i == 0) {
    out[1] = 1.0;
    *ticket = 0;
  }
}

__global__ void __launch_bounds__(TPB) k_pow_step(Csr<double> A, const double* __restrict__ dinv,
                                                  const double* __restrict__ xin, double* __restrict__ y,
                                                  double* partials, double* out /* lambda, scale */,
                                                  unsigned int* ticket) {
  __shared__ double sm[3][TPB / 32];
  __shared__ bool last;
  const double sc = out[1];
  double p[3] = {0.0, 0.0, 0.0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.nrows; i += gridDim.x * blockDim.x) {
    double ax = 0.0;
    for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) ax = fma(A.val[q], xin[A.col[q]] * sc, ax);
    const double di = dinv[i], xi = xin[i] * sc;
    p[0] = fma(xi, ax, p[0]);
    p[1] = fma(xi * xi, 1.0 / di, p[1]);
    p[2] = fma(ax * ax, di, p[2]);
    y[i] = di * ax;
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const auto warp_sums = [&]() {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) p[c] += __shfl_xor_sync(0xffffffffu, p[c], o);
      if (lane == 0) sm[c][w] = p[c];
    }
    __syncthreads();
  };
  warp_sums();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int k = 0; k < TPB / 32; ++k) t += sm[threadIdx.x][k];
    partials[3 * blockIdx.x + threadIdx.x] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    p[c] = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += TPB) p[c] += __ldcg(partials + 3 * b + c);
  }
  warp_sums();
  if (threadIdx.x == 0) {
    double t[3] = {0.0, 0.0, 0.0};
    for (int c = 0; c < 3; ++c)
      for (int k = 0; k < TPB / 32; ++k) t[c] += sm[c][k];
    out[0] = t[1] > 0.0 ? t[0] / t[1] : 0.0;
    out[1] = t[2] > 0.0 ? 1.0 / sqrt(t[2]) : 0.0;
    *ticket = 0;
  }
}

// lambda_max(D^-1 A) estimate (20 iterations) into out[0]; the caller caps it by the Gershgorin bound
static ch_status power_estimate(const Csr<double>& A, const double* dinv, cudaStream_t st, Alloc& tmp, double* out) {
  const int n = A.nrows;
  double *x = nullptr, *y = nullptr, *part = nullptr;
  unsigned int* ticket = nullptr;
  CH_TRY(tmp.get(&x, (size_t)n));
  CH_TRY(tmp.get(&y, (size_t)n));
  CH_TRY(tmp.get(&part, (size_t)3 * POW_BLOCKS));
  CH_TRY(tmp.get(&ticket, 1));
  const int nb = blocks_for(n) < POW_BLOCKS ? blocks_for(n) : POW_BLOCKS;
  k_pow_init<<<blocks_for(n), TPB, 0, st>>>(n, x, out, ticket);
  for (int it = 0; it < 20; ++it) {
    k_pow_step<<<nb, TPB, 0, st>>>(A, dinv, x, y, part, out, ticket);
    std::swap(x, y);
  }
  CH_LAUNCHED();
  return CH_OK;
}

// ---------------------------------------------------------------- set-up driver
static ch_status level_setup(Hierarchy* h, int l, const ch_params& p, cudaStream_t st, Alloc& ra,
                             bool* last) {
  const Csr<double>& A = h->A[l];
  const int n = A.nrows;
  double* dinv = nullptr;
  CH_TRY(h->mem.get(&dinv, (size_t)n));
  h->dinv.push_back(dinv);
  Alloc tmp;
  double *rb = nullptr, *est = nullptr;  // est: lambda estimate, its scale, the Gershgorin bound
  CH_TRY(tmp.get(&rb, (size_t)n));
  CH_TRY(tmp.get(&est, 3));
  CH_CUDA(cudaMemsetAsync(est, 0, 3 * sizeof(double), st));
  k_diag_gersh<<<blocks_for(n), TPB, 0, st>>>(A, dinv, rb);
  k_max_reduce<<<red_blocks(n), TPB, 0, st>>>(rb, n, reinterpret_cast<unsigned long long*>(est + 2));
  CH_LAUNCHED();
  CH_TRY(power_estimate(A, dinv, st, tmp, est));
  double h_est[3] = {0.0, 0.0, 0.0};
  CH_CUDA(cudaMemcpyAsync(h_est, est, sizeof(h_est), cudaMemcpyDeviceToHost, st));
  CH_CUDA(cudaStreamSynchronize(st));
  double rho = h_est[2];
  if (!(rho > 0.0) || !std::isfinite(rho)) {
    set_error("AMG level %d: bad Gershgorin bound %g (zero or non-finite diagonal?)", l, rho);
    return CH_ERR_NONFINITE;
  }
  // Gershgorin overestimates lambda_max(D^-1 A) on coarse aggregation levels (by 30-150% on the
  // meshes here), which would misplace the Chebyshev interval: use a power-iteration estimate
  // with a 5% margin, never above the Gershgorin bound.
  const double lam = h_est[0];
  if (lam > 0.0 && std::isfinite(lam)) rho = std::min(rho, 1.05 * lam);
  h->rho.push_back(rho);
  // coarse_max 0: 512 rows for FP64 V-cycles, 2048 for FP32 (where the dense inverse is half the
  // bytes); measured on 512 x 512, the dense solve beating the per-level launch chain up to there
  // (FP64: 512 and 1024 alike, 11.63 ms per step; FP32: 4.85-4.88 ms at 4096 rows, 4.75 at 2048;
  // the 64-run batch 30.9-31.1 ms either way, the 3D 128 x 128 x 32 box 14.8 ms either way)
  const int cmax = p.coarse_max > 0 ? p.coarse_max : (h->precision == 0 ? 512 : 2048);
  if (n <= cmax) {
    *last = true;
    return CH_OK;
  }
  // strength of connection
  uint8_t *s0 = nullptr, *s = nullptr;
  CH_TRY(tmp.get(&s0, (size_t)A.nnz));
  CH_TRY(tmp.get(&s, (size_t)A.nnz));
  int *skey = nullptr, *cnt = nullptr;
  double* sval = nullptr;  // entry scratch: normalised sizes here, the prolongator's coefficients below
  CH_TRY(tmp.get(&sval, (size_t)A.nnz));
  k_abs_diag<<<blocks_for(n), TPB, 0, st>>>(n, dinv, rb);
  k_strength<<<blocks_for(n), TPB, 0, st>>>(A, rb, p.amg_theta, sval, s0);
  k_strength_sym<<<blocks_for(n), TPB, 0, st>>>(A, s0, s);
  CH_LAUNCHED();
  // MIS(2)
  int8_t* state = nullptr;
  uint64_t *key = nullptr, *m1 = nullptr, *m2 = nullptr;
  int* und = nullptr;
  CH_TRY(tmp.get(&state, (size_t)n));
  CH_TRY(tmp.get(&key, (size_t)n));
  CH_TRY(tmp.get(&m1, (size_t)n));
  CH_TRY(tmp.get(&m2, (size_t)n));
  CH_TRY(tmp.get(&und, 1));
  CH_CUDA(cudaMemsetAsync(state, 1, (size_t)n, st));
  for (int round = 0;; ++round) {
    if (round > 70) {
      set_error("AMG level %d: MIS(2) did not finish", l);
      return CH_ERR_INTERNAL;
    }
    // three rounds between looks at the count of undecided nodes: a round after the last leaves the
    // states as they are, and costs less than the host's round trip
    for (int k = 0; k < 3; ++k) {
      k_mis_keys<<<blocks_for(n), TPB, 0, st>>>(n, state, key);
      k_strong_max<<<blocks_for(n), TPB, 0, st>>>(A, s, key, m1);
      k_strong_max<<<blocks_for(n), TPB, 0, st>>>(A, s, m1, m2);
      CH_CUDA(cudaMemsetAsync(und, 0, sizeof(int), st));
      k_mis_update<<<blocks_for(n), TPB, 0, st>>>(n, key, m2, state, und);
    }
    CH_LAUNCHED();
    int u = 0;
    CH_CUDA(cudaMemcpyAsync(&u, und, sizeof(int), cudaMemcpyDeviceToHost, st));
    CH_CUDA(cudaStreamSynchronize(st));
    if (u == 0) break;
  }
  // aggregates
  int *isroot = nullptr, *rootid = nullptr, *agg = nullptr, *agg2 = nullptr, *una = nullptr;
  CH_TRY(tmp.get(&isroot, (size_t)n));
  CH_TRY(tmp.get(&rootid, (size_t)n + 1));
  CH_TRY(tmp.get(&agg, (size_t)n));
  CH_TRY(tmp.get(&agg2, (size_t)n));
  CH_TRY(tmp.get(&una, 1));
  k_roots<<<blocks_for(n), TPB, 0, st>>>(n, state, isroot);
  CH_LAUNCHED();
  int64_t nc = 0;
  CH_TRY(scan_i32_to_rowptr(isroot, rootid, n, &nc, st, tmp));
  for (int pass = 0;; ++pass) {
    if (pass > 50) {
      set_error("AMG level %d: aggregation did not cover all nodes", l);
      return CH_ERR_INTERNAL;
    }
    // two passes per look (roots' neighbours, then theirs: MIS(2) usually needs no more); a pass over
    // assigned nodes copies
    for (int k = 0; k < 2; ++k) {
      CH_CUDA(cudaMemsetAsync(una, 0, sizeof(int), st));
      k_agg_pass<<<blocks_for(n), TPB, 0, st>>>(A, s, isroot, rootid, agg, agg2, pass == 0 && k == 0, una);
      std::swap(agg, agg2);
    }
    CH_LAUNCHED();
    int u = 0;
    CH_CUDA(cudaMemcpyAsync(&u, una, sizeof(int), cudaMemcpyDeviceToHost, st));
    CH_CUDA(cudaStreamSynchronize(st));
    if (u == 0) break;
  }
  // smoothed prolongator
  Csr<double> P;
  P.nrows = n;
  P.ncols = (int)nc;
  CH_TRY(tmp.get(&skey, (size_t)A.nnz));
  CH_TRY(tmp.get(&cnt, (size_t)n));
  const double omega = (4.0 / 3.0) / rho;
  k_prolong<false><<<blocks_for(n), TPB, 0, st>>>(A, dinv, agg, omega, skey, sval, cnt, nullptr,
                                                   nullptr, nullptr);
  CH_LAUNCHED();
  CH_TRY(h->mem.get(&P.rowptr, (size_t)n + 1));
  int64_t pnnz = 0;
  CH_TRY(scan_i32_to_rowptr(cnt, P.rowptr, n, &pnnz, st, tmp));
  P.nnz = pnnz;
  CH_TRY(h->mem.get(&P.col, (size_t)pnnz));
  CH_TRY(h->mem.get(&P.val, (size_t)pnnz));
  k_prolong<true><<<blocks_for(n), TPB, 0, st>>>(A, dinv, agg, omega, skey, sval, cnt, P.rowptr,
                                                  P.col, P.val);
  CH_LAUNCHED();
  Csr<double> R, AP, Ac;
  CH_TRY(transpose(P, &R, st, h->mem));
  Alloc aptmp;
  Csr<double> RA;
  if (h->precision == 1 && l > 0 && n <= 65536 && n >= 4 * nc && A.nnz <= 32LL * n) {
    // R A first: where it has no more entries than A, the cycle restricts by R b - (R A) x, one launch less and
    // no residual vector.  FP32 cycles below the finest level are bound by their launches (Algorithm 1, us per
    // application: 256 x 256 115.7 -> 108.5, 512 x 512 195.5 -> 183.6, 800 x 400 235 -> 220); FP64 ones by the
    // FP64 pipe (512 x 512 780 and 778), and larger levels by their entries (64 runs, 200000 rows: 942 -> 950).
    // Long rows of A (3D) or coarsening by less than 4 would give R A rows of thousands of entries.
    CH_TRY(spgemm(R, A, &RA, st, ra));
    CH_TRY(spgemm(RA, P, &Ac, st, h->mem));
    if (RA.nnz > A.nnz) RA = Csr<double>();
  } else {
    CH_TRY(spgemm(A, P, &AP, st, aptmp));
    CH_TRY(spgemm(R, AP, &Ac, st, h->mem));
  }
  h->P.push_back(P);
  h->R.push_back(R);
  h->A.push_back(Ac);
  h->RA.push_back(RA);
  CH_CUDA(cudaStreamSynchronize(st));
  return CH_OK;
}

template <typename T>
static ch_status tile_setup();
template <typename T, typename V2>
static void launch_residual(int tpr, const Csr<T>& A, const V2* b, const V2* x, V2* r, cudaStream_t st,
                            const LatOp<T>* lat = nullptr, bool pdl = false);
template <typename T, typename V2, bool ACC>
static void launch_spmv2(int tpr, const Csr<T>& A, const V2* x, V2* y, cudaStream_t st, bool pdl = false);
template <typename T, typename V2>
static void launch_restrict(const LevelT<T>& L, int tpr, const V2* x, V2* bc, const T* dinv, T invtheta, V2* xc,
                            cudaStream_t st, bool pdl);

// ---------------------------------------------------------------- SpMV tile autotuner
// Lanes per row (1..32, or a whole block for restrictions of long rows) for each matrix the V-cycle
// multiplies by: A (smoother steps and residuals), R (restriction), P (prolongation).  autotune = 0 takes the rule below; 1 times
// every candidate on the matrix itself (one warm-up, three timed launches) and keeps the rule's
// choice unless another is more than 5% faster.  Decisions are cached per process by matrix
// shape (kind, rows, columns, entries, value size), so rebuilding a hierarchy of the same shape
// reproduces its choices -- and its floating-point summation order -- exactly.  A process that
// wants its choices made on a busy GPU builds its first solver with autotune = 0 (nothing is
// cached then) and tunes afterwards.
static int tpr_rule(int64_t nnz, int rows) {
  const double avg = rows > 0 ? (double)nnz / rows : 1.0;
  int t = 1;
  while (t < 32 && 4.0 * t <= avg) t *= 2;
  return t;
}

static std::mutex g_tune_mu;
static std::map<std::tuple<int, int, int, int64_t, int>, int> g_tune_cache;

template <typename Launch>
static int tune_tpr(int kind, int rows, int cols, int64_t nnz, int tsize, int mode, Launch&& launch,
                    cudaStream_t st) {
  const int rule = tpr_rule(nnz, rows);
  if (mode == 0 || rows == 0) return rule;
  const auto key = std::make_tuple(kind, rows, cols, nnz, tsize);
  {
    std::lock_guard<std::mutex> lk(g_tune_mu);
    auto it = g_tune_cache.find(key);
    if (it != g_tune_cache.end()) return it->second;
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    cudaGetLastError();
    return rule;
  }
  // An idle GPU ramps its clocks over the first fraction of a second: warm up on the rule's width,
  // then time every width in two passes and keep each width's faster pass.
  // Restrictions with long rows also try a block per row.
  constexpr int NW = 7;
  const int width[NW] = {1, 2, 4, 8, 16, 32, 256};
  const int nw = kind == 1 && nnz >= 64LL * rows ? NW : NW - 1;
  for (int r = 0; r < 20; ++r) launch(rule);
  float t[NW];
  for (int k = 0; k < nw; ++k) t[k] = 1e30f;
  for (int pass = 0; pass < 2; ++pass) {
    for (int k = 0; k < nw; ++k) {
      const int tpr = width[k];
      launch(tpr);
      cudaEventRecord(e0, st);
      for (int r = 0; r < 3; ++r) launch(tpr);
      cudaEventRecord(e1, st);
      cudaEventSynchronize(e1);
      float ms = 1e30f;
      cudaEventElapsedTime(&ms, e0, e1);
      t[k] = std::min(t[k], ms);
    }
  }
  float best = 1e30f, t_rule = 1e30f;
  int pick = rule;
  for (int k = 0; k < nw; ++k) {
    if (width[k] == rule) t_rule = t[k];
    if (t[k] < best) {
      best = t[k];
      pick = width[k];
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaGetLastError();
  if (t_rule <= 1.05f * best) pick = rule;
  std::lock_guard<std::mutex> lk(g_tune_mu);
  g_tune_cache[key] = pick;
  return pick;
}

template <typename T>
static ch_status autotune_levels(Hierarchy* h, std::vector<LevelT<T>>& L, int mode, cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  for (int l = 0; l < h->nlev; ++l) {
    const int n = L[l].A.nrows;
    V2* vecs[4] = {L[l].x, L[l].x2, L[l].r, L[l].b};
    for (int k = 0; k < 4; ++k) CH_CUDA(cudaMemsetAsync(vecs[k], 0, sizeof(V2) * n, st));
  }
  for (int l = 0; l < h->nlev; ++l) {
    LevelT<T>& W = L[l];
    W.tprA = W.lat.nd ? 1
                      : tune_tpr(0, W.A.nrows, W.A.ncols, W.A.nnz, sizeof(T), mode,
                                 [&](int t) { launch_residual<T, V2>(t, W.A, W.b, W.x, W.r, st); }, st);
    if (l + 1 < h->nlev) {
      LevelT<T>& C = L[l + 1];
      const Csr<T>& R = W.RB.nnz > 0 ? W.RB : W.R;
      W.tprR = tune_tpr(1, R.nrows, R.ncols, R.nnz, sizeof(T), mode,
                        [&](int t) {
                          launch_restrict<T, V2>(W, t, W.x, C.b, (const T*)nullptr, T(0), (V2*)nullptr, st, false);
                        }, st);
      W.tprP = tune_tpr(2, W.P.nrows, W.P.ncols, W.P.nnz, sizeof(T), mode,
                        [&](int t) { launch_spmv2<T, V2, true>(t, W.P, C.x, W.x, st); }, st);
    }
  }
  CH_LAUNCHED();
  CH_CUDA(cudaStreamSynchronize(st));
  return CH_OK;
}

// Table rows of the lattice form from the representative nodes' CSR rows (slot nd: 1 / diagonal).
__global__ void k_lat_table(Csr<double> A, Lattice L, int nd, int ts, double* tab) {
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= L.nids) return;
  const int i = L.rep[id];
  const int2 w = L.wh[id];
  double* row = tab + (size_t)id * ts;
  for (int d = 0; d < ts; ++d) row[d] = 0.0;
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q)
    for (int d = 0; d < nd; ++d)
      if (lat_off(nd, d, w.x, w.y) == A.col[q] - i) row[d] = A.val[q];
  row[nd] = 1.0 / row[nd / 2];
}

// bad = 1 if a stored entry lies off its run's lattice stencil or further than `rel` of the diagonal from its
// class's table value
__global__ void k_lat_check(Csr<double> A, Lattice L, int nd, int ts, const double* tab, double rel, int* bad) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  const int id = lat_id(L, i);
  const int2 w = L.wh[id];
  const double* row = tab + (size_t)id * ts;
  const double tol = rel * fabs(row[nd / 2]);
  bool ok = true;
  unsigned seen = 0;
  for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) {
    int at = -1;
    for (int d = 0; d < nd; ++d)
      if (lat_off(nd, d, w.x, w.y) == A.col[q] - i) at = d;
    if (at < 0 || !(fabs(A.val[q] - row[at]) <= tol)) ok = false;
    if (at >= 0) seen |= 1u << at;
  }
  for (int d = 0; d < nd; ++d)
    if (!(seen >> d & 1) && row[d] != 0.0) ok = false;  // the class has an entry that the row lacks
  if (!ok) *bad = 1;
}

template <typename T>
__global__ void k_lat_cast(const double* a, T* b, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (T)a[i];
}

// The lattice form's FP64 table of A where every row fits it (tab stays null where not: the level
// then keeps the CSR form).
static ch_status lat_build(const Csr<double>& A, const Lattice* L, double rel, Alloc& mem, double** tab,
                           cudaStream_t st) {
  *tab = nullptr;
  const int nd = L->dim == 2 ? 7 : 15, ts = nd + 1;
  Alloc tmp;
  int* bad = nullptr;
  double* t = nullptr;
  CH_TRY(tmp.get(&bad, 1));
  CH_TRY(mem.get(&t, (size_t)L->nids * ts));
  CH_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), st));
  k_lat_table<<<blocks_for(L->nids), TPB, 0, st>>>(A, *L, nd, ts, t);
  k_lat_check<<<blocks_for(A.nrows), TPB, 0, st>>>(A, *L, nd, ts, t, rel, bad);
  CH_LAUNCHED();
  int hb = 0;
  CH_CUDA(cudaMemcpyAsync(&hb, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  CH_CUDA(cudaStreamSynchronize(st));
  if (!hb) *tab = t;
  return CH_OK;
}

// Coefficients of the Chebyshev smoother.  Step s from x with the carried direction e and r = A x - b:
//   e' = carry_s e + D^-1 r,  x' = x - beta_s e'
// (e is the usual direction d = x' - x over -beta: no factor per row is left).  The direction is kept rather
// than x - x_prev, which would feed x's rounding into the next steps (FP32 errors 3 to 24 % larger, FP64 ones
// 1.3 to 3.3 times with the diagonal folded as well).  A pass from zero starts with x = invtheta D^-1 b and
// its first step carries from_x x.
struct ChebCoef {
  double invtheta, from_x;
  double carry[16], beta[16];
};

// Tiles of a pass of `halo` operator applications over every run of a 2D mesh, none where a launch per step is
// faster.  FP32 block heights by the time they take in units of region rows, measured at degrees 1 to 16 over 256 x
// 256 .. 2048 x 2048, 800 x 400, 4000 x 60, 33 x 2000 and 16- and 64-run batches: a block alone on its SM costs its
// rows and 24 for its latencies, and as many waves as there are, so a mesh that fits one wave takes the shortest
// block that does; small halos on larger meshes take two blocks of 8 groups per SM, which overlap (a wave costs
// 62 and 10 per application -- a smaller region recomputes more -- and the last one only its share; vectors
// beyond L2 wait longer for their loads, and the overlap is worth more: 80).  Algorithm 1, us per application, two
// blocks / one: 1024 x 1024 degree 3 486 / 489, degree 8 726 / 685; 64 runs 909 / 926 and 1411 / 1308; 2048 x 2048
// 1655 / 1730 and 2496 / 2420.  Fewer than 4 groups are too few warps to hide anything.
// Tiles or steps: an application recomputes a tile's halo, so a step by tiles costs 1.3e-6 us per region node and a
// launch over the mesh 1.1 us and 5.9e-6 per node (1e-5 beyond L2), 2 us at least.  Times by tiles / by steps:
// 1024 x 1024 degree 5 546 / 714, 12 976 / 1159, 14 1255 / 1288, 15 1472 / 1357, 16 1754 / 1420; 64 runs degree 13
// 1911 / 1923, 16 3226 / 2214; 256 x 256 degree 16 266 / 381.
// FP64: the fewest region rows on the busiest SM.
template <typename T>
static ch_status tile_plan(const ch_mesh_s* m, int halo, Alloc& mem, TilePlan* out, cudaStream_t st) {
  using S = TileShape<T>;
  constexpr bool F32 = sizeof(T) == 4;
  *out = TilePlan();
  const int tw = S::RW - 2 * halo;
  if (tw < S::RW / 4) return CH_OK;
  const auto count = [&](int th) {
    int64_t n = 0;
    for (const ch_params& p : m->runs) n += (int64_t)((p.nx + tw) / tw) * ((p.ny + th) / th);
    return n;
  };
  const bool far = m->N > 3000000;  // four vectors and more of FP32 pairs do not fit L2
  double best = 0.0;
  int G = 0;
  bool pair = false;
  const auto consider = [&](int g, bool two) {
    const int rh = S::ROWS * g, th = rh - 2 * halo;
    if (th < 1 || S::RW * g % 32 != 0) return;
    const int64_t n = count(th);
    const double waves = (double)((n + 151) / 152);
    const double cost =
        two ? (far ? 80.0 : 62.0 + 10.0 * halo) * std::max(1.0, n / 304.0) : waves * (rh + (F32 ? 24 : 0));
    if (G == 0 || cost < best) {
      best = cost;
      G = g;
      pair = two;
    }
  };
  for (int g = F32 ? 4 : 2; g <= S::GMAX; ++g) consider(g, false);
  if (F32) consider(S::GPAIR, true);
  if (G == 0) return CH_OK;
  const int th = S::ROWS * G - 2 * halo;
  if (!F32 && count(th) > TILE_MAX_F64) return CH_OK;
  const double step = far ? 1e-5 * m->N : std::max(2.0, 1.1 + 5.9e-6 * m->N);
  if (F32 && 1.3e-6 * S::RW * S::ROWS * G * count(th) > step) return CH_OK;
  std::vector<LatTile> tiles;
  for (size_t r = 0; r < m->runs.size(); ++r) {
    const ch_params& p = m->runs[r];
    for (int y = 0; y <= p.ny; y += th)
      for (int x = 0; x <= p.nx; x += tw)
        tiles.push_back({m->run_off[r], p.nx + 1, p.ny + 1, x, y, (int)r * m->pos.ncls});
  }
  LatTile* d = nullptr;
  CH_TRY(mem.get(&d, tiles.size()));
  CH_CUDA(cudaMemcpyAsync(d, tiles.data(), sizeof(LatTile) * tiles.size(), cudaMemcpyHostToDevice, st));
  CH_CUDA(cudaStreamSynchronize(st));  // tiles is a host temporary
  out->ntiles = (int)tiles.size();
  out->groups = G;
  out->halo = halo;
  out->pair = pair;
  out->tiles = d;
  return CH_OK;
}

template <typename T>
static ch_status make_working(Hierarchy* h, const ch_mesh_s* mesh, std::vector<LevelT<T>>& L,
                              cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  L.resize(h->nlev);
  for (int l = 0; l < h->nlev; ++l) {
    LevelT<T>& w = L[l];
    auto cast_csr = [&](const Csr<double>& src, Csr<T>& dst) -> ch_status {
      dst.nrows = src.nrows;
      dst.ncols = src.ncols;
      dst.nnz = src.nnz;
      dst.rowptr = src.rowptr;
      dst.col = src.col;
      if (std::is_same<T, double>::value) {
        dst.val = reinterpret_cast<T*>(src.val);
      } else {
        CH_TRY(h->mem.get(&dst.val, (size_t)src.nnz));
        k_copy_cast<T><<<blocks_for(src.nnz), TPB, 0, st>>>(src.val, dst.val, src.nnz);
        CH_LAUNCHED();
      }
      return CH_OK;
    };
    CH_TRY(cast_csr(h->A[l], w.A));
    if (l + 1 < h->nlev) {
      CH_TRY(cast_csr(h->P[l], w.P));
      CH_TRY(cast_csr(h->R[l], w.R));
      if (h->RA[l].nnz > 0) {
        const Csr<double>&R = h->R[l], &RA = h->RA[l];
        w.RB.nrows = R.nrows;
        w.RB.ncols = R.ncols + RA.ncols;
        w.RB.nnz = R.nnz + RA.nnz;
        CH_TRY(h->mem.get(&w.RB.rowptr, (size_t)R.nrows + 1));
        CH_TRY(h->mem.get(&w.RB.col, (size_t)w.RB.nnz));
        CH_TRY(h->mem.get(&w.RB.val, (size_t)w.RB.nnz));
        k_stack<T><<<blocks_for(R.nrows, TPB / 32), TPB, 0, st>>>(R, RA, w.RB);
        CH_LAUNCHED();
      }
    }
    const int n = h->A[l].nrows;
    if (std::is_same<T, double>::value) {
      w.dinv = reinterpret_cast<T*>(h->dinv[l]);
    } else {
      CH_TRY(h->mem.get(&w.dinv, (size_t)n));
      k_copy_cast<T><<<blocks_for(n), TPB, 0, st>>>(h->dinv[l], w.dinv, n);
      CH_LAUNCHED();
    }
    CH_TRY(h->mem.get(&w.x, (size_t)n));
    CH_TRY(h->mem.get(&w.x2, (size_t)n));
    CH_TRY(h->mem.get(&w.r, (size_t)n));
    CH_TRY(h->mem.get(&w.b, (size_t)n));
    w.pdl = h->pdl;
  }

  // the fine level in lattice form (LatOp)
  constexpr bool F32 = sizeof(T) == 4;
  const Lattice* lat = F32 ? &mesh->pos : &mesh->lat;
  double* tab64 = nullptr;
  CH_TRY(lat_build(h->A[0], lat, F32 ? 0x1p-36 : 0.0, h->mem, &tab64, st));
  const bool by_position = F32 && tab64;
  if (F32 && !tab64) {
    lat = &mesh->lat;
    CH_TRY(lat_build(h->A[0], lat, 0.0, h->mem, &tab64, st));
  }
  if (tab64) {
    LatOp<T>& op = L[0].lat;
    op.nd = lat->dim == 2 ? 7 : 15;
    op.ts = op.nd + 1;
    op.L = *lat;
    const int cnt = lat->nids * op.ts;
    T* tab = nullptr;
    CH_TRY(h->mem.get(&tab, (size_t)cnt));
    k_lat_cast<T><<<blocks_for(cnt), TPB, 0, st>>>(tab64, tab, cnt);
    op.tab = tab;
    CH_LAUNCHED();
    if (lat->dim == 2 && h->nlev > 1 && (by_position || !F32)) {
      CH_TRY(tile_setup<T>());
      CH_TRY(tile_plan<T>(mesh, h->cheb_degree, h->mem, &L[0].plan, st));
      CH_TRY(tile_plan<T>(mesh, h->cheb_degree + 1, h->mem, &L[0].plan_r, st));
    }
  }
  return autotune_levels<T>(h, L, h->autotune, st);
}

ch_status hierarchy_build(const Csr<double>& A0, const ch_mesh_s* mesh, const ch_params& p, int precision, cudaStream_t st,
                          Hierarchy** out) {
  *out = nullptr;
  Hierarchy* h = new Hierarchy();
  h->precision = precision;
  h->cheb_degree = p.cheb_degree;
  // cheb_degree_coarse 0: degree 2 below the finest level (at most cheb_degree).  Measured on
  // 512 x 512 with the finest degree 5: FP64 79.8 / 75.9 / 70.9 and mixed 173.3 / 170.5 / 164.1
  // steps/s for coarse degrees 2 / 3 / 4
  h->cheb_degree_coarse = p.cheb_degree_coarse > 0 ? p.cheb_degree_coarse : std::min(2, p.cheb_degree);
  h->autotune = p.autotune;
  h->pdl = p.pdl != 0;
  h->cheb_lower = p.cheb_lower;
  h->A.push_back(A0);
  Alloc ra;  // the R A products, until the working copies hold them
  ch_status s = CH_OK;
  for (int l = 0;; ++l) {
    if (l >= 25) {
      set_error("AMG: more than 25 levels");
      s = CH_ERR_INTERNAL;
      break;
    }
    bool last = false;
    s = level_setup(h, l, p, st, ra, &last);
    if (s != CH_OK || last) break;
  }
  if (s == CH_OK) {
    h->nlev = (int)h->A.size();
    h->nc = h->A.back().nrows;
    if (h->nc > 4096) {
      set_error("AMG: coarsest level has %d rows (> 4096); coarsening stalled", h->nc);
      s = CH_ERR_INTERNAL;
    }
  }
  if (s == CH_OK) {
    Alloc tmp;
    double* D = nullptr;
    int* bad = nullptr;
    const int nc = h->nc;
    double *R = nullptr, *L = nullptr;
    s = tmp.get(&bad, 1);
    if (s == CH_OK) s = tmp.get(&R, (size_t)GJ_B * nc);
    if (s == CH_OK) s = tmp.get(&L, (size_t)GJ_B * nc);
    if (s == CH_OK) s = h->mem.get(&h->cinv, (size_t)nc * nc);
    if (s == CH_OK) {
      D = h->cinv;  // inverted in place
      cudaMemsetAsync(bad, 0, sizeof(int), st);
      cudaMemsetAsync(D, 0, sizeof(double) * (size_t)nc * nc, st);
      k_to_dense<<<blocks_for(nc), TPB, 0, st>>>(h->A.back(), D);
      const int nt = (nc + GJ_B - 1) / GJ_B;
      for (int k0 = 0; k0 < nc; k0 += GJ_B) {
        k_gj_panel<<<nt, 256, 0, st>>>(nc, k0, D, R, L, bad);
        k_gj_update<<<dim3(nt, nt), 256, 0, st>>>(nc, k0, D, R, L);
      }
      int hb = 0;
      cudaMemcpyAsync(&hb, bad, sizeof(int), cudaMemcpyDeviceToHost, st);
      if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
        set_error("AMG: coarse inverse failed");
        s = CH_ERR_CUDA;
      } else if (hb) {
        set_error("AMG: coarsest operator not positive definite");
        s = CH_ERR_INTERNAL;
      }
    }
  }
  if (s == CH_OK) {
    if (precision == 0) {
      s = make_working<double>(h, mesh, h->Ld, st);
    } else {
      s = make_working<float>(h, mesh, h->Lf, st);
      if (s == CH_OK) s = h->mem.get(&h->cinvf, (size_t)h->nc * h->nc);
      if (s == CH_OK) {
        k_d2f<<<blocks_for((int64_t)h->nc * h->nc), TPB, 0, st>>>(h->cinv, h->cinvf,
                                                                  (int64_t)h->nc * h->nc);
      }
    }
    if (s == CH_OK && cudaStreamSynchronize(st) != cudaSuccess) {
      set_error("AMG: building working copies failed");
      s = CH_ERR_CUDA;
    }
    h->RA.clear();
  }
  if (s != CH_OK) {
    delete h;
    return s;
  }
  *out = h;
  return CH_OK;
}

void hierarchy_free(Hierarchy* h) { delete h; }
int hierarchy_levels(const Hierarchy* h) { return h ? h->nlev : 0; }
void hierarchy_level_tiles(const Hierarchy* h, int l, int* tA, int* tR, int* tP) {
  const int a = h->precision == 0 ? h->Ld[l].tprA : h->Lf[l].tprA;
  const int r = h->precision == 0 ? h->Ld[l].tprR : h->Lf[l].tprR;
  const int q = h->precision == 0 ? h->Ld[l].tprP : h->Lf[l].tprP;
  if (tA) *tA = a;
  if (tR) *tR = l + 1 < h->nlev ? r : 0;
  if (tP) *tP = l + 1 < h->nlev ? q : 0;
}

void hierarchy_level_size(const Hierarchy* h, int l, int64_t* rows, int64_t* nnz) {
  if (rows) *rows = h->A[l].nrows;
  if (nnz) *nnz = h->A[l].nnz;
}

// Level l as the V-cycle uses it: the FP64 set-up matrices A_l and P_l (device to device copies
// into caller buffers), the Chebyshev interval [cheb_lower, 1] x 1.1 rho_l of D^-1 A_l and the
// smoothing degree; the coarsest level has no P and no smoothing (dense inverse).
ch_status hierarchy_level_export(const Hierarchy* h, int l, int64_t* rows, int64_t* nnz, int64_t* nnz_P,
                                 double* lo, double* hi, int* degree, int* A_rowptr, int* A_col,
                                 double* A_val, int* P_rowptr, int* P_col, double* P_val, cudaStream_t st) {
  const Csr<double>& A = h->A[l];
  const bool coarsest = l + 1 == h->nlev;
  const int64_t np = coarsest ? 0 : h->P[l].nnz;
  if (rows) *rows = A.nrows;
  if (nnz) *nnz = A.nnz;
  if (nnz_P) *nnz_P = np;
  const double top = coarsest ? 0.0 : 1.1 * h->rho[l];
  if (hi) *hi = top;
  if (lo) *lo = h->cheb_lower * top;
  if (degree) *degree = coarsest ? 0 : (l == 0 ? h->cheb_degree : h->cheb_degree_coarse);
  const auto copy = [&](void* dst, const void* src, size_t bytes) -> ch_status {
    if (dst && bytes) CH_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, st));
    return CH_OK;
  };
  CH_TRY(copy(A_rowptr, A.rowptr, sizeof(int) * ((size_t)A.nrows + 1)));
  CH_TRY(copy(A_col, A.col, sizeof(int) * (size_t)A.nnz));
  CH_TRY(copy(A_val, A.val, sizeof(double) * (size_t)A.nnz));
  if (!coarsest) {
    const Csr<double>& P = h->P[l];
    CH_TRY(copy(P_rowptr, P.rowptr, sizeof(int) * ((size_t)P.nrows + 1)));
    CH_TRY(copy(P_col, P.col, sizeof(int) * (size_t)P.nnz));
    CH_TRY(copy(P_val, P.val, sizeof(double) * (size_t)P.nnz));
  }
  return CH_OK;
}

// ---------------------------------------------------------------- V-cycle kernels (2 RHS)
// When a V-cycle kernel lets its successor be scheduled (programmatic dependent launch): right
// after its dependency wait in FP32, where the kernels are short and bound by latency, so the
// successor's blocks are resident when it finishes; not at all in FP64, where the kernels are
// bound by the FP64 pipe and successor blocks that arrive early crowd the SMs unevenly.  Measured
// on the 512 x 512 mesh, ms per time step: FP32 V-cycles 8.33 plain, 8.06 without the trigger,
// 7.96 with it; FP64 V-cycles 16.90 plain, 16.78 without, 17.70 with it (16.75 when only grids of
// at most 152 blocks trigger, 17.28 at most 608; that small-grid rule took FP64 32 x 32 steps from
// 2.26 to 2.21 ms but 128 x 128 steps from 2.95 to 3.03).
template <typename T>
__device__ __forceinline__ void pdl_trigger_t() {
  if (sizeof(T) == 4) pdl_trigger();
}

template <typename T, typename V2>
__device__ __forceinline__ V2 mk2(T a, T b) {
  V2 v;
  v.x = a;
  v.y = b;
  return v;
}

// x = D^-1 b / theta (first Chebyshev step from a zero guess)
template <typename T, typename V2>
__global__ void k_cheb_first(int n, const T* dinv, const V2* b, T invtheta, V2* x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const T di = i < n ? dinv[i] : T(0);  // set-up data: read before the dependency wait
  pdl_wait();
  pdl_trigger_t<T>();
  if (i >= n) return;
  const T s = invtheta * di;
  const V2 bi = b[i];
  x[i] = mk2<T, V2>(s * bi.x, s * bi.y);
}

// Row sums of A x for both right-hand sides with TPR lanes per row: lane `sub` takes entries
// sub, sub+TPR, ... of the row and shuffles add the lanes' partial sums in a fixed order.  The two sums
// are separated in the first round (each half of the lanes keeps one and takes the other half's part of
// it), so they cost log2 TPR additions and not twice as many, and what follows a row sum runs in two
// lanes, one per right-hand side: an FP64 instruction holds the SM's pipe 16 clocks however few lanes it
// serves (Algorithm 1 per application, us: FP64 800 x 400 1049 -> 993, 63 x 47 x 41 2105 -> 1710 with
// k_restrict_wide; FP32 128 x 128 x 32 960 -> 882).  Threads past the last row contribute zeros (no early return before the shuffles).  The
// sum adds onto the caller's (s0, s1), which lane 0 of a row may seed (with -b: the sum is then A x - b at
// no extra FP64 instruction).
//
// The row's structure and values are set-up data, so a kernel reads them before its programmatic
// dependency wait (row_prefetch: the lane's first CsrRow::PF entries, i.e. rowptr, then val and col)
// and only gathers x after it (row_acc): one dependent L2 round trip behind the wait instead of
// three (rowptr, col, x).  Entries past the prefetched ones are read after the wait, in the same
// order.
template <typename T, int TPR>
struct CsrRow {
  static constexpr int PF = TPR == 1 ? 8 : (TPR <= 4 ? 4 : 2);  // entries per lane read early
  int q = 0, e = 0;  // the lane's next entry after the prefetched ones; the row's end
  T a[PF];
  int c[PF];
};

template <typename T, int TPR>
__device__ __forceinline__ void row_prefetch(const Csr<T>& A, int row, int sub, CsrRow<T, TPR>& r) {
  constexpr int PF = CsrRow<T, TPR>::PF;
#pragma unroll
  for (int k = 0; k < PF; ++k) {
    r.a[k] = T(0);
    r.c[k] = -1;
  }
  if (row < A.nrows) {
    const int b = A.rowptr[row] + sub;
    r.e = A.rowptr[row + 1];
#pragma unroll
    for (int k = 0; k < PF; ++k) {
      const int q = b + k * TPR;
      if (q < r.e) {
        r.a[k] = A.val[q];
        r.c[k] = A.col[q];
      }
    }
    r.q = b + PF * TPR;
  }
}

// What a matrix multiplies: a vector, or two stacked ones (n entries of b, then x).
template <typename V2>
struct OneVec {
  const V2* __restrict__ x;
  __device__ __forceinline__ V2 operator[](int c) const { return x[c]; }
};
template <typename V2>
struct TwoVecs {
  const V2* __restrict__ b;
  const V2* __restrict__ x;
  int n;
  __device__ __forceinline__ V2 operator[](int c) const { return c < n ? b[c] : x[c - n]; }
};

template <typename T, typename V2, int TPR, typename X>
__device__ __forceinline__ void row_acc(const Csr<T>& A, const CsrRow<T, TPR>& r, const X& x, T& s0, T& s1) {
  constexpr int PF = CsrRow<T, TPR>::PF;
  V2 xj[PF];
#pragma unroll
  for (int k = 0; k < PF; ++k)
    if (r.c[k] >= 0) xj[k] = x[r.c[k]];
#pragma unroll
  for (int k = 0; k < PF; ++k)
    if (r.c[k] >= 0) {
      s0 = fma(r.a[k], xj[k].x, s0);
      s1 = fma(r.a[k], xj[k].y, s1);
    }
#pragma unroll 4
  for (int q = r.q; q < r.e; q += TPR) {
    const T a = A.val[q];
    const V2 v = x[A.col[q]];
    s0 = fma(a, v.x, s0);
    s1 = fma(a, v.y, s1);
  }
}

// The row sums over the TPR lanes of a row: component 0 in the row's lane 0, component 1 in its lane
// TPR / 2 (TPR = 1: both in the one lane).
template <typename T, int TPR>
struct RowSum {
  T v[TPR == 1 ? 2 : 1];
};
template <typename T, int TPR>
__device__ __forceinline__ RowSum<T, TPR> row_sum(T s0, T s1, int sub) {
  RowSum<T, TPR> r;
  r.v[0] = s0;
  if constexpr (TPR == 1) {
    r.v[1] = s1;
  } else {
    constexpr int H = TPR / 2;
    const bool up = sub & H;
    const T send = up ? s0 : s1;
    T keep = up ? s1 : s0;
    keep += __shfl_xor_sync(0xffffffffu, send, H);
#pragma unroll
    for (int o = H / 2; o > 0; o >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, o);
    r.v[0] = keep;
  }
  return r;
}
// f(component, sum) in the lanes that hold a row's sums
template <typename T, int TPR, typename F>
__device__ __forceinline__ void row_finish(const RowSum<T, TPR>& r, int sub, F f) {
  if constexpr (TPR == 1) {
    f(0, r.v[0]);
    f(1, r.v[1]);
  } else {
    constexpr int H = TPR / 2;
    if ((sub & (H - 1)) == 0) f(sub != 0, r.v[0]);  // (TPR = 2: H - 1 = 0, both lanes)
  }
}
template <typename V2> __device__ __forceinline__ auto* comps(V2* p) { return &p->x; }
template <typename V2> __device__ __forceinline__ const auto* comps(const V2* p) { return &p->x; }

// One Chebyshev step (ChebCoef); the row sum starts from -b.  `from`: what the direction carries on from;
// keep: the next step of the pass reads it.
enum Carry { CARRY_NONE = 0, CARRY_E = 1, CARRY_X = 2 };  // nothing; e; x (the pass's first iterate, from zero)
template <typename T, typename V2, int TPR>
__global__ void __launch_bounds__(TPB) k_cheb_step(Csr<T> A, const T* __restrict__ dinv,
                                                   const V2* __restrict__ b, const V2* __restrict__ x,
                                                   V2* __restrict__ xo, V2* __restrict__ e, T carry, T nbeta,
                                                   int from, bool keep) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = t / TPR, sub = t % TPR;
  CsrRow<T, TPR> row;
  row_prefetch<T, TPR>(A, i, sub, row);
  const T di = i < A.nrows ? dinv[i] : T(0);
  pdl_wait();
  pdl_trigger_t<T>();
  T s0 = 0, s1 = 0;
  if (sub == 0 && i < A.nrows) {
    const V2 bi = b[i];
    s0 = -bi.x;
    s1 = -bi.y;
  }
  row_acc<T, V2, TPR>(A, row, OneVec<V2>{x}, s0, s1);
  const RowSum<T, TPR> r = row_sum<T, TPR>(s0, s1, sub);
  if (i >= A.nrows) return;
  row_finish<T, TPR>(r, sub, [&](int c, T s) {
    const T y = comps(x + i)[c];
    T v = di * s;
    if (from != CARRY_NONE) v = fma(carry, from == CARRY_E ? comps(e + i)[c] : y, v);
    if (keep) comps(e + i)[c] = v;
    comps(xo + i)[c] = fma(nbeta, v, y);
  });
}

template <typename T, typename V2, int TPR>
__global__ void __launch_bounds__(TPB) k_residual(Csr<T> A, const V2* __restrict__ b,
                                                  const V2* __restrict__ x, V2* __restrict__ r) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = t / TPR, sub = t % TPR;
  CsrRow<T, TPR> row;
  row_prefetch<T, TPR>(A, i, sub, row);
  pdl_wait();
  pdl_trigger_t<T>();
  T s0 = 0, s1 = 0;
  row_acc<T, V2, TPR>(A, row, OneVec<V2>{x}, s0, s1);
  const RowSum<T, TPR> rs = row_sum<T, TPR>(s0, s1, sub);
  if (i >= A.nrows) return;
  row_finish<T, TPR>(rs, sub, [&](int c, T s) { comps(r + i)[c] = comps(b + i)[c] - s; });
}

// y = A x (ACC = false) or y += A x (ACC = true)
template <typename T, typename V2, int TPR, bool ACC, typename X>
__global__ void __launch_bounds__(TPB) k_spmv2(Csr<T> A, X x, V2* __restrict__ y) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = t / TPR, sub = t % TPR;
  CsrRow<T, TPR> row;
  row_prefetch<T, TPR>(A, i, sub, row);
  pdl_wait();
  pdl_trigger_t<T>();
  T s0 = 0, s1 = 0;
  row_acc<T, V2, TPR>(A, row, x, s0, s1);
  const RowSum<T, TPR> rs = row_sum<T, TPR>(s0, s1, sub);
  if (i >= A.nrows) return;
  row_finish<T, TPR>(rs, sub, [&](int c, T s) {
    T* o = comps(y + i) + c;
    *o = ACC ? *o + s : s;
  });
}

// ---------------------------------------------------------------- structured (lattice) fine level
// One row of the lattice form: the class's ND values and factor and its run's strides (set-up data, so
// the kernels read them before their dependency wait).  Rows of a warp are of one class by position,
// of two to four by inexact widths: the table reads are broadcasts from L1.
template <typename T, int ND>
struct LatRow {
  T a[ND + 1];
  int W, WH;
};
// a table row in 16-byte loads (rows are 32 to 128 bytes, aligned to their size), value by value into o
template <int N>
__device__ __forceinline__ void load_table_row(const float* __restrict__ src, float (&o)[N]) {
#pragma unroll
  for (int q = 0; q < N / 4; ++q) {
    const float4 v = reinterpret_cast<const float4*>(src)[q];
    o[4 * q] = v.x;
    o[4 * q + 1] = v.y;
    o[4 * q + 2] = v.z;
    o[4 * q + 3] = v.w;
  }
}
template <int N>
__device__ __forceinline__ void load_table_row(const double* __restrict__ src, double (&o)[N]) {
#pragma unroll
  for (int q = 0; q < N / 2; ++q) {
    const double2 v = reinterpret_cast<const double2*>(src)[q];
    o[2 * q] = v.x;
    o[2 * q + 1] = v.y;
  }
}
template <typename T, int ND>
__device__ __forceinline__ LatRow<T, ND> lat_row(const LatOp<T>& D, const T* __restrict__ tab, int i) {
  LatRow<T, ND> r;
  const int id = lat_id(D.L, i);
  r.W = D.L.W;
  r.WH = D.L.WH;
  if (D.L.multi) {
    const int2 w = D.L.wh[id];
    r.W = w.x;
    r.WH = w.y;
  }
  load_table_row(tab + (size_t)id * (ND + 1), r.a);
  return r;
}

// Row sum of the lattice form onto the caller's (s0, s1) (zero, or -b for a residual's negative).
template <typename T, typename V2, int ND>
__device__ __forceinline__ void lat_row_acc(const LatRow<T, ND>& r, int n, int i, const V2* __restrict__ x,
                                            T& s0, T& s1) {
#pragma unroll
  for (int d = 0; d < ND; ++d) {
    int j = i + lat_off(ND, d, r.W, r.WH);
    j = j < 0 ? 0 : (j >= n ? n - 1 : j);
    const V2 xj = x[j];
    s0 = fma(r.a[d], xj.x, s0);
    s1 = fma(r.a[d], xj.y, s1);
  }
}

// One Chebyshev step on the lattice form: k_cheb_step's arithmetic.  FP32 is bound by its vectors (42 bytes
// per row: x, b, e read and written, x' and the class id; one value per stored entry as well made it 72 in 2D,
// 104 in 3D), FP64 by its pipe (ten instructions per right-hand side in 2D).  FP32 128 x
// 128 x 32 8.7 us, FP64 512 x 512 11.8.
template <typename T, typename V2, int ND>
__global__ void __launch_bounds__(TPB) k_cheb_step_lat(LatOp<T> D, int n, const V2* __restrict__ b,
                                                       const V2* __restrict__ x, V2* __restrict__ xo,
                                                       V2* __restrict__ e, T carry, T nbeta, int from, bool keep) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  LatRow<T, ND> row;
  if (i < n) row = lat_row<T, ND>(D, D.tab, i);
  pdl_wait();
  pdl_trigger_t<T>();
  if (i >= n) return;
  const V2 bi = b[i];
  T s0 = -bi.x, s1 = -bi.y;
  lat_row_acc<T, V2, ND>(row, n, i, x, s0, s1);
  const V2 y = x[i];
  V2 v = mk2<T, V2>(row.a[ND] * s0, row.a[ND] * s1);
  if (from != CARRY_NONE) {
    const V2 d = from == CARRY_E ? e[i] : y;
    v = mk2<T, V2>(fma(carry, d.x, v.x), fma(carry, d.y, v.y));
  }
  if (keep) e[i] = v;
  xo[i] = mk2<T, V2>(fma(nbeta, v.x, y.x), fma(nbeta, v.y, y.y));
}

template <typename T, typename V2, int ND>
__global__ void __launch_bounds__(TPB) k_residual_lat(LatOp<T> D, int n, const V2* __restrict__ b,
                                                      const V2* __restrict__ x, V2* __restrict__ r) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  LatRow<T, ND> row;
  if (i < n) row = lat_row<T, ND>(D, D.tab, i);
  pdl_wait();
  pdl_trigger_t<T>();
  if (i >= n) return;
  T s0 = 0, s1 = 0;
  lat_row_acc<T, V2, ND>(row, n, i, x, s0, s1);
  const V2 bi = b[i];
  r[i] = mk2<T, V2>(bi.x - s0, bi.y - s1);
}

template <typename T, typename V2, int ND>
__global__ void __launch_bounds__(TPB) k_spmv2_lat(LatOp<T> D, int n, const V2* __restrict__ x, V2* __restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  LatRow<T, ND> row;
  if (i < n) row = lat_row<T, ND>(D, D.tab, i);
  pdl_wait();
  pdl_trigger_t<T>();
  if (i >= n) return;
  T s0 = 0, s1 = 0;
  lat_row_acc<T, V2, ND>(row, n, i, x, s0, s1);
  y[i] = mk2<T, V2>(s0, s1);
}

// A whole smoothing pass of the 2D lattice form in one launch.  A block holds a region of RW columns x
// (ROWS x groups) rows: a tile of outputs and a halo as deep as the pass applies the operator
// (deg times), in shared memory (two buffers of the iterate); a thread owns ROWS nodes of one column
// with their iterate, the direction and b in registers.  Every application spoils one ring of the
// region, so the tile's own nodes end exact: the same operations in the same order as k_cheb_step_lat
// and k_residual_lat, bitwise.  Operators being one table row per class, nothing but b (and x, unless
// the pass starts from zero) is read, once per pass instead of four vectors per step.
//   ZERO: the pass starts from a zero guess (its first step is pointwise);  RES: r = b - A x' as well.
// Nodes outside the mesh stay zero (their coefficients are zero).
// Bound by the latencies of a block's loads and steps, not memory.  Algorithm 1 per application, us, one
// launch per step -> per pass: FP32 64 x 64 141 -> 67, 256 x 256 183 -> 118, 512 x 512 268 -> 197, 1024 x
// 1024 695 -> 532, 64 runs 1138 -> 969; FP64 32 x 32 146 -> 90, 64 x 64 214 -> 164.
template <typename T, typename V2>
struct TileArgs {
  const LatTile* tiles;
  const T* tab;  // the operator's table
  const V2 *b, *x;
  V2 *xo, *r;
  double* wo;  // the last pass of an application: the result goes here in FP64, ldw values per node, not to xo
  Lattice L;   // FP64: the nodes' class ids
  int ldw, deg, halo;
  T invtheta, carry[16], nbeta[16];
};
template <typename T>
constexpr int tile_smem(int groups) {
  return 2 * (TileShape<T>::ROWS * groups + 3) * (TileShape<T>::RW + 2) * 2 * (int)sizeof(T);
}

// a x + y and the like on both right-hand sides: packed FP32 (one instruction for two fused
// multiply-adds, each rounded as fmaf), plain FP64
__device__ __forceinline__ unsigned long long pk2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 up2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ float2 fma2(float c, float2 x, float2 a) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pk2(c, c)), "l"(pk2(x.x, x.y)), "l"(pk2(a.x, a.y)));
  return up2(r);
}
__device__ __forceinline__ float2 mul2(float c, float2 x) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk2(c, c)), "l"(pk2(x.x, x.y)));
  return up2(r);
}
__device__ __forceinline__ double2 fma2(double c, double2 x, double2 a) {
  return make_double2(fma(c, x.x, a.x), fma(c, x.y, a.y));
}
__device__ __forceinline__ double2 mul2(double c, double2 x) { return make_double2(c * x.x, c * x.y); }

// One block's tile.  FP64: a thread's one node has its class's row (by cell widths).  FP32 (classes by
// position): a thread's nodes share the column's row, and those of the first and last mesh row load theirs.
// EDGE: the region reaches the mesh's boundary (or past it), and nodes outside the mesh stay zero; the other
// tiles (all but the rim) test nothing.
template <typename T, typename V2, bool ZERO, bool RES, bool EDGE>
__device__ __forceinline__ void smooth_tile(const TileArgs<T, V2>& a, const LatTile& tl, V2* buf) {
  constexpr int RW = TileShape<T>::RW, ROWS = TileShape<T>::ROWS, ST = RW + 2;
  const int tid = threadIdx.x, c = tid % RW, g = tid / RW, RH = ROWS * (blockDim.x / RW);
  const int plane = (RH + 3) * ST;  // node (r, c) of a buffer at (r + 1, c + 1)
  const int h = a.halo, x = tl.x0 - h + c, y0 = tl.y0 - h + g * ROWS;
  const bool col_in = !EDGE || (x >= 0 && x < tl.W);
  const int cx = !EDGE ? 1 : (x <= 0 ? 0 : (x >= tl.W - 1 ? 2 : 1));
  const auto in = [&](int t) { return !EDGE || (col_in && (unsigned)(y0 + t) < (unsigned)tl.H); };
  const size_t node0 = (size_t)tl.off + (size_t)((long long)y0 * tl.W) + x;  // (used only inside the mesh)
  constexpr bool OWN = ROWS == 1;  // the thread has one node, with its own row
  const int own = OWN && in(0) ? lat_id(a.L, (int)node0) : 0;
  const auto load_row = [&](const T* tab, int cy, T (&o)[8]) {
    load_table_row(tab + (size_t)(OWN ? own : tl.id0 + cx + 3 * cy) * 8, o);
  };
  const auto edge = [&](int t) { return y0 + t == 0 ? 0 : (y0 + t == tl.H - 1 ? 2 : 1); };
  T row[8];
  load_row(a.tab, 1, row);
  pdl_wait();
  pdl_trigger_t<T>();
  V2 nb[ROWS], cur[ROWS], dir[ROWS];  // -b, the iterate and the direction (ChebCoef's e)
#pragma unroll
  for (int t = 0; t < ROWS; ++t) {
    nb[t] = cur[t] = dir[t] = mk2<T, V2>(T(0), T(0));
    if (in(t)) {
      const V2 bt = a.b[node0 + (size_t)t * tl.W];
      nb[t] = mk2<T, V2>(-bt.x, -bt.y);
      if (!ZERO) cur[t] = a.x[node0 + (size_t)t * tl.W];
    }
  }
  if (ZERO) {
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      T di = row[7];
      if (EDGE && !OWN && edge(t) != 1) {
        T e[8];
        load_row(a.tab, edge(t), e);
        di = e[7];
      }
      const T s = -(a.invtheta * di);
      dir[t] = cur[t] = mk2<T, V2>(s * nb[t].x, s * nb[t].y);  // (carry[1] is ChebCoef's from_x)
    }
  }
  V2* mine = buf + (g * ROWS + 1) * ST + c + 1;  // this thread's first node in buffer 0
#pragma unroll
  for (int t = 0; t < ROWS; ++t) mine[t * ST] = cur[t];
  __syncthreads();
  int p = 0, margin = 0;
  // f(t, 1 / diagonal, sum) for the thread's nodes, sum = the operator applied to the iterate, seeded with -b
  // or 0 (the thread's row, or the interior one of its column, is in `row`)
  const auto apply = [&](bool seed_b, auto f) {
    const V2* q = mine + p * plane;
    V2 south = q[-ST], wprev = q[-ST - 1], wcur = q[-1], ecur = q[1], enext = q[ST + 1];
#pragma unroll
    for (int t = 0; t < ROWS; ++t) {
      const V2 north = t + 1 < ROWS ? cur[t + 1 < ROWS ? t + 1 : t] : q[ROWS * ST];
      const V2 center = cur[t];
      const int r = g * ROWS + t;
      if (r > margin && r < RH - 1 - margin && in(t)) {
        V2 s = seed_b ? nb[t] : mk2<T, V2>(T(0), T(0));
        const V2 nbr[7] = {wprev, south, wcur, center, ecur, north, enext};
        if (EDGE && !OWN && edge(t) != 1) {
          T e[8];
          load_row(a.tab, edge(t), e);
#pragma unroll
          for (int d = 0; d < 7; ++d) s = fma2(e[d], nbr[d], s);
          f(t, e[7], s);
        } else {
#pragma unroll
          for (int d = 0; d < 7; ++d) s = fma2(row[d], nbr[d], s);
          f(t, row[7], s);
        }
      }
      south = center;
      wprev = wcur;
      wcur = q[(t + 1) * ST - 1];
      ecur = enext;
      enext = q[(t + 2) * ST + 1];
    }
    ++margin;
  };
  for (int s = ZERO ? 1 : 0; s < a.deg; ++s) {
    const T carry = a.carry[s], nbeta = a.nbeta[s];
    apply(true, [&](int t, T dinv, V2 sum) {
      dir[t] = fma2(carry, dir[t], mul2(dinv, sum));
      cur[t] = fma2(nbeta, dir[t], cur[t]);
    });
    p ^= 1;
#pragma unroll
    for (int t = 0; t < ROWS; ++t) mine[p * plane + t * ST] = cur[t];
    __syncthreads();
  }
  const bool col_out = col_in && c >= h && c < RW - h;
  const auto out = [&](int t) { return col_out && in(t) && g * ROWS + t >= h && g * ROWS + t < RH - h; };
#pragma unroll
  for (int t = 0; t < ROWS; ++t)
    if (out(t)) {
      const size_t i = node0 + (size_t)t * tl.W;
      if (!ZERO && !RES && a.wo)
        *reinterpret_cast<double2*>(a.wo + i * a.ldw) = make_double2((double)cur[t].x, (double)cur[t].y);
      else
        a.xo[i] = cur[t];
    }
  if (RES) {
    apply(false, [&](int t, T, V2 sum) {
      if (out(t)) a.r[node0 + (size_t)t * tl.W] = mk2<T, V2>(-nb[t].x - sum.x, -nb[t].y - sum.y);
    });
  }
}

// PAIR: two blocks per SM (64 registers a thread in FP32; the single blocks take up to 80 and spill nothing)
template <typename T, typename V2, bool ZERO, bool RES, bool PAIR>
__global__ void __launch_bounds__(TileShape<T>::RW*(PAIR ? TileShape<T>::GPAIR : TileShape<T>::GMAX), PAIR ? 2 : 1)
    k_smooth_tile(TileArgs<T, V2> a) {
  extern __shared__ __align__(16) unsigned char tile_raw[];
  V2* buf = reinterpret_cast<V2*>(tile_raw);
  const LatTile tl = a.tiles[blockIdx.x];
  constexpr int RW = TileShape<T>::RW, ROWS = TileShape<T>::ROWS;
  const int RH = ROWS * (blockDim.x / RW), xl = tl.x0 - a.halo, yl = tl.y0 - a.halo;
  if (xl > 0 && yl > 0 && xl + RW < tl.W && yl + RH < tl.H) smooth_tile<T, V2, ZERO, RES, false>(a, tl, buf);
  else smooth_tile<T, V2, ZERO, RES, true>(a, tl, buf);
}

#define CH_LAT_DISPATCH(nd, KCALL)                    \
  switch (nd) {                                       \
    case 7: { constexpr int NDC = 7; KCALL; } break;  \
    default: { constexpr int NDC = 15; KCALL; } break; \
  }

// b_c = R r (or R b - R A x), fused with the coarse level's first Chebyshev step from a zero guess
// (pointwise: x_c = invtheta D_c^-1 b_c, the arithmetic of k_cheb_first): one launch instead of two.
template <typename T, typename V2, int TPR, typename X>
__global__ void __launch_bounds__(TPB) k_restrict_first(Csr<T> R, X r, V2* __restrict__ bc,
                                                        const T* __restrict__ dinv_c, T invtheta,
                                                        V2* __restrict__ xc) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = t / TPR, sub = t % TPR;
  CsrRow<T, TPR> row;
  row_prefetch<T, TPR>(R, i, sub, row);
  const T f = i < R.nrows ? invtheta * dinv_c[i] : T(0);
  pdl_wait();
  pdl_trigger_t<T>();
  T s0 = 0, s1 = 0;
  row_acc<T, V2, TPR>(R, row, r, s0, s1);
  const RowSum<T, TPR> rs = row_sum<T, TPR>(s0, s1, sub);
  if (i >= R.nrows) return;
  row_finish<T, TPR>(rs, sub, [&](int c, T s) {
    comps(bc + i)[c] = s;
    comps(xc + i)[c] = f * s;
  });
}

// A restriction whose rows are long and few (the coarsest levels of a 3D hierarchy: 443 rows of 700
// entries gave 443 warps, 17.8 us in FP32 and 32.6 in FP64, now 8.2 in FP64): one block per row.  FIRST:
// fused with the coarse level's first Chebyshev step as k_restrict_first.  Chosen by the set-up's timing
// (WIDE lanes per row).
constexpr int WIDE = TPB;
template <typename T, typename V2, bool FIRST, typename X>
__global__ void __launch_bounds__(TPB) k_restrict_wide(Csr<T> R, X r, V2* __restrict__ bc,
                                                       const T* __restrict__ dinv_c, T invtheta,
                                                       V2* __restrict__ xc) {
  __shared__ T part[2][TPB / 32];
  const int i = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  CsrRow<T, WIDE> row;
  row_prefetch<T, WIDE>(R, i, threadIdx.x, row);
  const T f = FIRST ? invtheta * dinv_c[i] : T(0);
  pdl_wait();
  pdl_trigger_t<T>();
  T s0 = 0, s1 = 0;
  row_acc<T, V2, WIDE>(R, row, r, s0, s1);
  const RowSum<T, 32> rs = row_sum<T, 32>(s0, s1, lane);
  if ((lane & 15) == 0) part[lane >> 4][w] = rs.v[0];
  __syncthreads();
  if (threadIdx.x < 2) {
    T s = part[threadIdx.x][0];
#pragma unroll
    for (int q = 1; q < TPB / 32; ++q) s += part[threadIdx.x][q];
    comps(bc + i)[threadIdx.x] = s;
    if (FIRST) comps(xc + i)[threadIdx.x] = f * s;
  }
}

#define CH_TPR_DISPATCH(tpr, KCALL)                      \
  switch (tpr) {                                         \
    case 1: { constexpr int TPRC = 1; KCALL; } break;    \
    case 2: { constexpr int TPRC = 2; KCALL; } break;    \
    case 4: { constexpr int TPRC = 4; KCALL; } break;    \
    case 8: { constexpr int TPRC = 8; KCALL; } break;    \
    case 16: { constexpr int TPRC = 16; KCALL; } break;  \
    default: { constexpr int TPRC = 32; KCALL; } break;  \
  }

// one Chebyshev step on a CSR level
template <typename T, typename V2>
static void launch_cheb_step(int tpr, const Csr<T>& A, const T* dinv, const V2* b, const V2* x, V2* xo,
                             V2* e, T carry, T nbeta, int from, bool keep, cudaStream_t st, bool pdl) {
  const int g = blocks_for((int64_t)A.nrows * tpr);
  CH_TPR_DISPATCH(tpr, (launch_k(pdl, k_cheb_step<T, V2, TPRC>, g, TPB, 0, st, A, dinv, b, x, xo, e, carry,
                                 nbeta, from, keep)));
}
template <typename T, typename V2>
static void launch_residual(int tpr, const Csr<T>& A, const V2* b, const V2* x, V2* r, cudaStream_t st,
                            const LatOp<T>* lat, bool pdl) {
  if (lat && lat->nd) {
    const int g = blocks_for(A.nrows);
    CH_LAT_DISPATCH(lat->nd, (launch_k(pdl, k_residual_lat<T, V2, NDC>, g, TPB, 0, st, *lat, A.nrows, b, x, r)));
    return;
  }
  const int g = blocks_for((int64_t)A.nrows * tpr);
  CH_TPR_DISPATCH(tpr, (launch_k(pdl, k_residual<T, V2, TPRC>, g, TPB, 0, st, A, b, x, r)));
}
// y = A x with the level's operator (the lattice form where there is one)
template <typename T, typename V2>
static void launch_apply_level(const LevelT<T>& L, const V2* x, V2* y, cudaStream_t st) {
  if (L.lat.nd) {
    const int g = blocks_for(L.A.nrows);
    CH_LAT_DISPATCH(L.lat.nd, (launch_k(L.pdl, k_spmv2_lat<T, V2, NDC>, g, TPB, 0, st, L.lat, L.A.nrows, x, y)));
    return;
  }
  launch_spmv2<T, V2, false>(L.tprA, L.A, x, y, st, L.pdl);
}
template <typename T, typename V2, bool ACC>
static void launch_spmv2(int tpr, const Csr<T>& A, const V2* x, V2* y, cudaStream_t st, bool pdl) {
  const int g = blocks_for((int64_t)A.nrows * tpr);
  CH_TPR_DISPATCH(tpr, (launch_k(pdl, k_spmv2<T, V2, TPRC, ACC, OneVec<V2>>, g, TPB, 0, st, A, OneVec<V2>{x}, y)));
}

// bc = R x, and with dinv the coarse level's first step from zero, xc = invtheta D^-1 bc
template <typename T, typename V2, typename X>
static void launch_restrict_x(int tpr, const Csr<T>& R, const X& x, V2* bc, const T* dinv, T invtheta, V2* xc,
                              cudaStream_t st, bool pdl) {
  const int g = blocks_for((int64_t)R.nrows * tpr);
  if (tpr == WIDE) {
    if (dinv) launch_k(pdl, k_restrict_wide<T, V2, true, X>, R.nrows, TPB, 0, st, R, x, bc, dinv, invtheta, xc);
    else launch_k(pdl, k_restrict_wide<T, V2, false, X>, R.nrows, TPB, 0, st, R, x, bc, dinv, invtheta, xc);
  } else if (dinv) {
    CH_TPR_DISPATCH(tpr, (launch_k(pdl, k_restrict_first<T, V2, TPRC, X>, g, TPB, 0, st, R, x, bc, dinv, invtheta,
                                   xc)));
  } else {
    CH_TPR_DISPATCH(tpr, (launch_k(pdl, k_spmv2<T, V2, TPRC, false, X>, g, TPB, 0, st, R, x, bc)));
  }
}
// a level's restriction: R r, or [R, -R A] (b, x) where it has the product
template <typename T, typename V2>
static void launch_restrict(const LevelT<T>& L, int tpr, const V2* x, V2* bc, const T* dinv, T invtheta, V2* xc,
                            cudaStream_t st, bool pdl) {
  if (L.RB.nnz > 0)
    launch_restrict_x<T, V2>(tpr, L.RB, TwoVecs<V2>{L.b, x, L.A.nrows}, bc, dinv, invtheta, xc, st, pdl);
  else
    launch_restrict_x<T, V2>(tpr, L.R, OneVec<V2>{L.r}, bc, dinv, invtheta, xc, st, pdl);
}

// x = Ainv b, dense nc x nc.  WPR warps per row: lane l of the row's warp `sub` takes columns
// sub * 32 + l + k * 32 WPR, with its first U entries of Ainv read before the dependency wait and
// 8 loads in flight after it; the lanes' sums are added as in row_sum and the warps' in warp order.
template <typename T, typename V2, int WPR>
__global__ void __launch_bounds__(TPB) k_dense_solve(int n, const T* __restrict__ inv, const V2* __restrict__ b,
                                                     V2* __restrict__ x) {
  static_assert((TPB / 32) % WPR == 0, "a row's warps share a block");
  constexpr int U = 8;  // the lane's first entries, read before the dependency wait
  __shared__ T part[TPB / 32][2];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int row = gw / WPR, sub = gw % WPR;
  const bool on = row < n;
  const int stride = 32 * WPR, j0 = sub * 32 + lane;
  const T* __restrict__ a = inv + (size_t)(on ? row : 0) * n;
  T pa[U];
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const int j = j0 + k * stride;
    pa[k] = (on && j < n) ? a[j] : T(0);
  }
  pdl_wait();
  pdl_trigger_t<T>();
  T s0 = 0, s1 = 0;
  if (on) {
    V2 bj[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int j = j0 + k * stride;
      if (j < n) bj[k] = b[j];
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (j0 + k * stride < n) {
        s0 = fma(pa[k], bj[k].x, s0);
        s1 = fma(pa[k], bj[k].y, s1);
      }
    }
#pragma unroll 8
    for (int j = j0 + U * stride; j < n; j += stride) {
      const T aj = a[j];
      const V2 v = b[j];
      s0 = fma(aj, v.x, s0);
      s1 = fma(aj, v.y, s1);
    }
  }
  T t = row_sum<T, 32>(s0, s1, lane).v[0];  // component 0 in lane 0, 1 in lane 16
  if ((lane & 15) == 0) part[w][lane >> 4] = t;
  __syncthreads();
  if (on && sub == 0 && (lane & 15) == 0) {
#pragma unroll
    for (int q = 1; q < WPR; ++q) t += part[w + q][lane >> 4];
    comps(x + row)[lane >> 4] = t;
  }
}

// x = Ainv b on the dense coarsest level, two warps per row.  Measured alone with the inverse
// flushed from L2 (us per solve, one / two / four warps per row): 3742 FP32 rows 26.2 / 22.5 / 24.8,
// 2048 FP32 rows 14.3 / 9.8 / 10.5, 512 FP64 rows 11.1 / 7.8 / 9.8.
template <typename T, typename V2>
static void launch_dense_solve(bool pdl, int n, const T* cinv, const V2* b, V2* x, cudaStream_t st) {
  launch_k(pdl, k_dense_solve<T, V2, 2>, blocks_for((int64_t)n * 64), TPB, 0, st, n, cinv, b, x);
}

// fine-level I/O: strided fp64 pairs <-> working precision pairs
template <typename T, typename V2>
__global__ void k_load2(int n, const double* src, int ld, V2* dst) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  pdl_trigger_t<T>();
  if (i >= n) return;
  const double2 v = *reinterpret_cast<const double2*>(src + (size_t)i * ld);
  dst[i] = mk2<T, V2>((T)v.x, (T)v.y);
}
// k_load2 fused with the finest level's first Chebyshev step from a zero guess (the arithmetic of
// k_cheb_first on the converted values): b = (T) src, x = invtheta D^-1 b.  One launch instead
// of two at the start of the first V-cycle of a solve.
template <typename T, typename V2>
__global__ void k_load2_first(int n, const double* src, int ld, const T* dinv, T invtheta, V2* b, V2* x) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const T di = i < n ? dinv[i] : T(0);  // set-up data: read before the dependency wait
  pdl_wait();
  pdl_trigger_t<T>();
  if (i >= n) return;
  const double2 v = *reinterpret_cast<const double2*>(src + (size_t)i * ld);
  const V2 bi = mk2<T, V2>((T)v.x, (T)v.y);
  b[i] = bi;
  const T s = invtheta * di;
  x[i] = mk2<T, V2>(s * bi.x, s * bi.y);
}
template <typename T, typename V2>
__global__ void k_store2(int n, const V2* src, double* dst, int ld) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  pdl_trigger_t<T>();
  if (i >= n) return;
  const V2 v = src[i];
  *reinterpret_cast<double2*>(dst + (size_t)i * ld) = make_double2((double)v.x, (double)v.y);
}

// ---------------------------------------------------------------- V-cycle driver
// Coefficients of `deg` Chebyshev semi-iteration steps for eigenvalues in [lo, hi]: the first
// step from zero is x = D^-1 b / theta, then d = alpha_s d + beta_s D^-1 (b - A x), x += d, kept as ChebCoef
// says.
static ChebCoef cheb_coef_interval(double lo, double hi, int deg) {
  ChebCoef c{};
  const double theta = 0.5 * (hi + lo), delta = 0.5 * (hi - lo), sigma = theta / delta;
  c.invtheta = 1.0 / theta;
  c.beta[0] = 1.0 / theta;
  double rho_prev = 1.0 / sigma;
  for (int s = 1; s < deg && s < 16; ++s) {
    const double r = 1.0 / (2.0 * sigma - rho_prev);
    const double alpha = r * rho_prev;
    c.beta[s] = 2.0 * r / delta;
    c.carry[s] = alpha * c.beta[s - 1] / c.beta[s];
    if (s == 1) c.from_x = -alpha / c.beta[1];
    rho_prev = r;
  }
  return c;
}

// the V-cycle smoother's interval: [lower, 1] x 1.1 rho
static ChebCoef cheb_coef(double rho, int deg, double lower) {
  const double hi = 1.1 * rho;
  return cheb_coef_interval(lower * hi, hi, deg);
}

static int semi_steps(const ch_params& p) { return p.cheb_M_steps > 0 ? p.cheb_M_steps : 5; }
// Wathen's bounds of the eigenvalues of D^-1 M: [1/2, 2] (triangles), [1/2, 5/2] (tetrahedra)
static ChebCoef semi_coef(int dim, int steps) { return cheb_coef_interval(0.5, dim == 2 ? 2.0 : 2.5, steps); }

// the tile kernels' shared-memory limits (above the 48 KB default)
template <typename T>
static ch_status tile_setup() {
  using V2 = typename V2T<T>::t;
  const auto set = [](auto kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, tile_smem<T>(TileShape<T>::GMAX));
  };
  CH_CUDA(set(k_smooth_tile<T, V2, true, true, false>));
  CH_CUDA(set(k_smooth_tile<T, V2, false, true, false>));
  CH_CUDA(set(k_smooth_tile<T, V2, false, false, false>));
  if constexpr (sizeof(T) == 4) {
    CH_CUDA(set(k_smooth_tile<T, V2, true, true, true>));
    CH_CUDA(set(k_smooth_tile<T, V2, false, true, true>));
    CH_CUDA(set(k_smooth_tile<T, V2, false, false, true>));
  }
  return CH_OK;
}

// the V-cycle smoother's pass on the finest level in one launch (see k_smooth_tile)
template <typename T, bool ZERO, bool RES>
static void launch_smooth_tile(const Hierarchy* h, LevelT<T>& L, const typename V2T<T>::t* x,
                               typename V2T<T>::t* xo, cudaStream_t st, double* wo = nullptr, int ldw = 0) {
  using V2 = typename V2T<T>::t;
  const TilePlan& pl = RES && !ZERO ? L.plan_r : L.plan;
  const ChebCoef c = cheb_coef(h->rho[0], h->cheb_degree, h->cheb_lower);
  TileArgs<T, V2> a;
  a.tiles = pl.tiles;
  a.tab = L.lat.tab;
  a.b = L.b;
  a.x = x;
  a.xo = xo;
  a.r = L.r;
  a.wo = wo;
  a.ldw = ldw;
  a.L = L.lat.L;
  a.deg = h->cheb_degree;
  a.halo = pl.halo;
  a.invtheta = (T)c.invtheta;
  for (int s = 0; s < 16; ++s) {
    a.carry[s] = (T)(ZERO && s == 1 ? c.from_x : c.carry[s]);
    a.nbeta[s] = (T)-c.beta[s];
  }
  const double n = L.A.nrows, apps = pl.halo;
  ProfScope ps(st, K_CHEB_STEP, sizeof(T) == 4,
               n * (2.0 * sizeof(T) * ((ZERO ? 1 : 2) + (RES ? 2 : (wo ? 0 : 1))) + (wo ? 16.0 : 0.0)),
               apps * (2.0 * L.A.nnz + 6.0 * n));
  const int threads = TileShape<T>::RW * pl.groups, smem = tile_smem<T>(pl.groups);
  if constexpr (sizeof(T) == 4) {
    if (pl.pair) {
      launch_k(L.pdl, k_smooth_tile<T, V2, ZERO, RES, true>, pl.ntiles, threads, smem, st, a);
      return;
    }
  }
  launch_k(L.pdl, k_smooth_tile<T, V2, ZERO, RES, false>, pl.ntiles, threads, smem, st, a);
}

// bytes per row of the fine level's lattice form beyond its vectors: the class id
static double lat_bytes(const Lattice& L, double n) { return (L.id32 ? 4.0 : 2.0) * n; }

// `deg` Chebyshev steps with coefficients c on level L (accounted as kernels kfirst / kstep), the direction in
// L.r (the residual's place, free while a level smooths).  zero_guess: 0 continue from *xcur; 1 start from
// zero (the first step is pointwise); 2 start from zero with that first step already taken by the
// caller (fused into the restriction or the input conversion)
template <typename T_>
static ch_status smooth_coef(LevelT<T_>& L, const ChebCoef& c, int deg, int zero_guess, int kfirst,
                             int kstep, typename V2T<T_>::t** xcur, cudaStream_t st) {
  using V2 = typename V2T<T_>::t;
  const int n = L.A.nrows;
  V2* x = *xcur;
  V2* other = (x == L.x) ? L.x2 : L.x;
  int s0 = 0;
  const double T = sizeof(T_), nnz = (double)L.A.nnz;
  if (zero_guess == 1) {
    ProfScope ps(st, kfirst, sizeof(T_) == 4, 5.0 * T * n, 2.0 * n);
    launch_k(L.pdl, k_cheb_first<T_, V2>, blocks_for(n), TPB, 0, st, n, L.dinv, L.b, (T_)c.invtheta, x);
    s0 = 1;
  } else if (zero_guess == 2) {
    s0 = 1;
  }
  // operator bytes: CSR values + column indices + row pointers and D^-1, or the class ids
  const double opb = L.lat.nd ? lat_bytes(L.lat.L, n) : nnz * (4 + T) + 4.0 * (n + 1) + T * n;
  for (int s = s0; s < deg; ++s) {
    const int from = s == 0 ? CARRY_NONE : (s == 1 && s0 == 1 ? CARRY_X : CARRY_E);
    const bool keep = s + 1 < deg;
    const T_ carry = (T_)(from == CARRY_X ? c.from_x : c.carry[s]), nbeta = (T_)-c.beta[s];
    ProfScope ps(st, kstep, sizeof(T_) == 4, opb + T * n * (6 + (from == CARRY_E ? 2 : 0) + (keep ? 2 : 0)),
                 2.0 * nnz + 6.0 * n);
    if (L.lat.nd) {
      CH_LAT_DISPATCH(L.lat.nd, (launch_k(L.pdl, k_cheb_step_lat<T_, V2, NDC>, blocks_for(n), TPB, 0, st, L.lat, n,
                                          L.b, x, other, L.r, carry, nbeta, from, keep)));
    } else {
      launch_cheb_step<T_, V2>(L.tprA, L.A, L.dinv, L.b, x, other, L.r, carry, nbeta, from, keep, st, L.pdl);
    }
    std::swap(x, other);
  }
  CH_LAUNCHED();
  *xcur = x;
  return CH_OK;
}

// the V-cycle's smoother on level l: its degree and interval
template <typename T_>
static ch_status smooth(Hierarchy* h, LevelT<T_>& L, int l, int zero_guess,
                        typename V2T<T_>::t** xcur, cudaStream_t st) {
  const int deg = l == 0 ? h->cheb_degree : h->cheb_degree_coarse;
  const ChebCoef c = cheb_coef(h->rho[l], deg, h->cheb_lower);
  return smooth_coef<T_>(L, c, deg, zero_guess, l == 0 ? K_CHEB_FIRST : K_CHEB_FIRST_C,
                         l == 0 ? K_CHEB_STEP : K_CHEB_STEP_C, xcur, st);
}

// M~^-1 by the Chebyshev semi-iteration (Section 3's alternative to AMG for the mass matrix):
// `steps` steps on D^-1 M from a zero guess over Wathen's bounds of its eigenvalues for P1
// simplices (semi_coef), on the finest level of M's hierarchy (its working-precision copy of M and
// D^-1).  b in L.b; result in *xres.
template <typename T_>
static ch_status semi_iteration(LevelT<T_>& L, int dim, int steps, typename V2T<T_>::t** xres, cudaStream_t st) {
  *xres = L.x;
  return smooth_coef<T_>(L, semi_coef(dim, steps), steps, 1, K_CHEB_SEMI, K_CHEB_SEMI, xres, st);
}

// one V-cycle at level l on L[l].b; result in *xres (L[l].x or L[l].x2).  zero_guess: as smooth_coef
// the level's smoothing passes run as tiles
template <typename T>
static bool tiled(const LevelT<T>& L) {
  return L.plan.ntiles > 0 && L.plan_r.ntiles > 0;
}

// (wo, ldw): where the finest level is tiled, the last pass stores the result there in FP64 (see TileArgs) and
// no conversion follows: Algorithm 1, us per application, 512 x 512 182.4 -> 180.0, 64 runs 940 -> 921
template <typename T>
static ch_status vcycle(Hierarchy* h, LevelT<T>* Ls, const T* cinv, int l,
                        int zero_guess, typename V2T<T>::t** xres, cudaStream_t st, double* wo = nullptr,
                        int ldw = 0) {
  using V2 = typename V2T<T>::t;
  LevelT<T>& L = Ls[l];
  const int n = L.A.nrows;
  const double Tb = sizeof(T);
  if (l == h->nlev - 1) {
    ProfScope ps(st, K_COARSE, sizeof(T) == 4, Tb * n * (double)n + 4.0 * Tb * n, 2.0 * n * (double)n);
    launch_dense_solve<T, V2>(L.pdl, n, cinv, L.b, L.x, st);
    CH_LAUNCHED();
    *xres = L.x;
    return CH_OK;
  }
  V2* x = *xres;
  LevelT<T>& C = Ls[l + 1];
  const int nc = C.A.nrows;
  const bool tiles = l == 0 && tiled(L);
  if (tiles) {
    V2* to = x == L.x ? L.x2 : L.x;
    if (zero_guess) launch_smooth_tile<T, true, true>(h, L, nullptr, to, st);
    else launch_smooth_tile<T, false, true>(h, L, x, to, st);
    CH_LAUNCHED();
    x = to;
  } else {
    CH_TRY(smooth<T>(h, L, l, zero_guess, &x, st));
    if (L.RB.nnz == 0) {
      const double opb = L.lat.nd ? lat_bytes(L.lat.L, n) : L.A.nnz * (4 + Tb) + 4.0 * (n + 1);
      ProfScope ps(st, l == 0 ? K_VRESIDUAL : K_VRESIDUAL_C, sizeof(T) == 4, opb + 6.0 * Tb * n, 2.0 * L.A.nnz);
      launch_residual<T, V2>(L.tprA, L.A, L.b, x, L.r, st, &L.lat, L.pdl);
    }
  }
  const bool fuse = l + 1 < h->nlev - 1;  // the coarse level smooths: fuse its first step
  {
    const Csr<T>& R = L.RB.nnz > 0 ? L.RB : L.R;
    ProfScope ps(st, l == 0 ? K_RESTRICT : K_RESTRICT_C, sizeof(T) == 4,
                 R.nnz * (4 + Tb) + 4.0 * (nc + 1) + 2.0 * Tb * (R.ncols + nc) + (fuse ? 3.0 * Tb * nc : 0.0),
                 2.0 * R.nnz + (fuse ? 2.0 * nc : 0.0));
    const T invtheta = (T)cheb_coef(h->rho[l + 1], h->cheb_degree_coarse, h->cheb_lower).invtheta;
    launch_restrict<T, V2>(L, L.tprR, x, C.b, fuse ? C.dinv : nullptr, invtheta, C.x, st, L.pdl);
  }
  CH_LAUNCHED();
  V2* xc = C.x;
  CH_TRY(vcycle<T>(h, Ls, cinv, l + 1, fuse ? 2 : 1, &xc, st));
  {
    ProfScope ps(st, l == 0 ? K_PROLONG : K_PROLONG_C, sizeof(T) == 4,
                 L.P.nnz * (4 + Tb) + 4.0 * (n + 1) + 2.0 * Tb * nc + 4.0 * Tb * n, 2.0 * L.P.nnz);
    launch_spmv2<T, V2, true>(L.tprP, L.P, xc, x, st, L.pdl);
  }
  CH_LAUNCHED();
  if (tiles) {
    V2* to = x == L.x ? L.x2 : L.x;
    launch_smooth_tile<T, false, false>(h, L, x, to, st, wo, ldw);
    CH_LAUNCHED();
    x = to;
  } else {
    CH_TRY(smooth<T>(h, L, l, 0, &x, st));
  }
  *xres = x;
  return CH_OK;
}

template <typename T>
static ch_status solve_t(Hierarchy* h, LevelT<T>* Ls, const T* cinv, const double* b,
                         int ldb, double* x, int ldx, int ncyc, cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  LevelT<T>& L = Ls[0];
  const int n = L.A.nrows;
  launch_k(L.pdl, k_load2<T, V2>, blocks_for(n), TPB, 0, st, n, b, ldb, L.b);
  CH_LAUNCHED();
  V2* xr = L.x;
  for (int c = 0; c < ncyc; ++c) CH_TRY(vcycle<T>(h, Ls, cinv, 0, c == 0, &xr, st));
  launch_k(L.pdl, k_store2<T, V2>, blocks_for(n), TPB, 0, st, n, xr, x, ldx);
  CH_LAUNCHED();
  return CH_OK;
}

// `passes` passes of the finest level's Chebyshev smoother of degree `degree` (the V-cycle's
// interval), each continuing from the previous pass's x; x (N x 2, fp64) is read and overwritten
template <typename T>
static ch_status smooth_t(Hierarchy* h, std::vector<LevelT<T>>& Ls, const double* b, double* x, int degree,
                          int passes, cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  LevelT<T>& L = Ls[0];
  const int n = L.A.nrows;
  const double io = n * (16.0 + 2.0 * sizeof(T));
  const ChebCoef c = cheb_coef(h->rho[0], degree, h->cheb_lower);
  {
    ProfScope ps(st, K_VLOAD, sizeof(T) == 4, 2.0 * io, 0.0);
    launch_k(L.pdl, k_load2<T, V2>, blocks_for(n), TPB, 0, st, n, b, 2, L.b);
  }
  {
    ProfScope ps(st, K_VLOAD, sizeof(T) == 4, 0.0, 0.0);  // its bytes are counted with the first load
    launch_k(L.pdl, k_load2<T, V2>, blocks_for(n), TPB, 0, st, n, x, 2, L.x);
  }
  CH_LAUNCHED();
  V2* xr = L.x;
  for (int k = 0; k < passes; ++k)
    CH_TRY(smooth_coef<T>(L, c, degree, 0, K_CHEB_FIRST, K_CHEB_STEP, &xr, st));
  {
    ProfScope ps(st, K_VSTORE, sizeof(T) == 4, io, 0.0);
    launch_k(L.pdl, k_store2<T, V2>, blocks_for(n), TPB, 0, st, n, xr, x, 2);
  }
  CH_LAUNCHED();
  return CH_OK;
}

ch_status hierarchy_smooth(Hierarchy* h, const double* b, double* x, int degree, int passes, cudaStream_t st) {
  if (h->precision == 0) return smooth_t<double>(h, h->Ld, b, x, degree, passes, st);
  return smooth_t<float>(h, h->Lf, b, x, degree, passes, st);
}

ch_status hierarchy_solve(Hierarchy* h, const double* b, int ldb, double* x, int ldx, int ncyc,
                          cudaStream_t st) {
  if (h->precision == 0) return solve_t<double>(h, h->Ld.data(), h->cinv, b, ldb, x, ldx, ncyc, st);
  return solve_t<float>(h, h->Lf.data(), h->cinvf, b, ldb, x, ldx, ncyc, st);
}

// ---------------------------------------------------------------- Algorithm 1
// w_1 = AMG(M) v_1;  w_2 = AMG(H) v_2;  w_2 = M w_2;  w_2 = AMG(H) w_2.
// v, w are N x 4 (phi_p, phi_n, mu_p, mu_n per node): block 1 at offset 0, block 2 at offset 2.
// The fine-level input of a solve: b = (T) v (strided FP64 pairs).  With AMG V-cycles on a
// hierarchy of more than one level the first V-cycle's first smoothing step (from zero) is done in
// the same launch (k_load2_first), and the V-cycle then starts at its second step (zero_guess 2).
// Returns the zero_guess for the first V-cycle.
template <typename T>
static int load_input(Hierarchy* h, LevelT<T>& L, bool amg, const double* v, int ld, cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  const int n = L.A.nrows;
  if (amg && h->nlev > 1 && !(L.plan.ntiles > 0 && L.plan_r.ntiles > 0)) {
    const ChebCoef c = cheb_coef(h->rho[0], h->cheb_degree, h->cheb_lower);
    ProfScope ps(st, K_VLOAD, sizeof(T) == 4, n * (16.0 + 5.0 * sizeof(T)), 2.0 * n);
    launch_k(L.pdl, k_load2_first<T, V2>, blocks_for(n), TPB, 0, st, n, v, ld, L.dinv, (T)c.invtheta, L.b, L.x);
    return 2;
  }
  ProfScope ps(st, K_VLOAD, sizeof(T) == 4, n * (16.0 + 2.0 * sizeof(T)), 0.0);
  launch_k(L.pdl, k_load2<T, V2>, blocks_for(n), TPB, 0, st, n, v, ld, L.b);
  return 1;
}

template <typename T>
static ch_status precond_t(ch_precond_s* pc, std::vector<LevelT<T>>& LM, std::vector<LevelT<T>>& LH,
                           const T* cinvM, const T* cinvH, const double* v, double* w,
                           cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  const int n = LM[0].A.nrows;
  const ch_params& p = pc->sys->p;
  // Step 1 does not depend on steps 2-4: it runs on the preconditioner's side stream, forked
  // from and joined back into st (inside a stream capture this becomes two parallel graph
  // branches).  Both chains are mostly latency-bound coarse-level launches, so they overlap.
  // With per-launch event timing on, everything stays on st so that kernel times do not overlap.
  const bool fork = pc->side != nullptr && !prof_timing();
  cudaStream_t sm = st;
  if (fork) {
    CH_CUDA(cudaEventRecord(pc->ev_fork, st));
    CH_CUDA(cudaStreamWaitEvent(pc->side, pc->ev_fork, 0));
    sm = pc->side;
  }
  // step 1: M w_1 = v_1 (w_1 in columns 0-1 of w; steps 2-4 write columns 2-3)
  {
    LevelT<T>& L = LM[0];
    const int zg = load_input<T>(pc->hM, L, p.precond_M != 1, v, 4, sm);
    V2* xr = L.x;
    if (p.precond_M == 1) {
      CH_TRY(semi_iteration<T>(L, pc->sys->mesh->dim, semi_steps(p), &xr, sm));
    } else {
      for (int c = 0; c < p.vcycles_M; ++c)
        CH_TRY(vcycle<T>(pc->hM, LM.data(), cinvM, 0, c == 0 ? zg : 0, &xr, sm, c + 1 == p.vcycles_M ? w : nullptr, 4));
    }
    if (p.precond_M == 1 || !tiled(L)) {
      ProfScope ps(sm, K_VSTORE, sizeof(T) == 4, n * (16.0 + 2.0 * sizeof(T)), 0.0);
      launch_k(L.pdl, k_store2<T, V2>, blocks_for(n), TPB, 0, sm, n, xr, w, 4);
    }
    CH_LAUNCHED();
  }
  if (fork) CH_CUDA(cudaEventRecord(pc->ev_join, sm));
  // steps 2-4: H w_2 = v_2; w_2 = M w_2; H w_2 = w_2
  {
    LevelT<T>& L = LH[0];
    const int zg = load_input<T>(pc->hH, L, true, v + 2, 4, st);
    V2* xr = L.x;
    for (int c = 0; c < p.vcycles_H; ++c) CH_TRY(vcycle<T>(pc->hH, LH.data(), cinvH, 0, c == 0 ? zg : 0, &xr, st));
    // b <- M x (M's fine level in working precision); the V-cycle reads only L.b afterwards
    {
      const double Tb = sizeof(T), nnz = (double)LM[0].A.nnz;
      const double opb = LM[0].lat.nd ? lat_bytes(LM[0].lat.L, n) : nnz * (4 + Tb) + 4.0 * (n + 1);
      ProfScope ps(st, K_SPMV_M, sizeof(T) == 4, opb + 4.0 * Tb * n, 2.0 * nnz);
      launch_apply_level<T, V2>(LM[0], xr, L.b, st);
    }
    CH_LAUNCHED();
    xr = L.x;  // the first solve's result now lives in L.b as M x; start afresh
    for (int c = 0; c < p.vcycles_H; ++c)
      CH_TRY(vcycle<T>(pc->hH, LH.data(), cinvH, 0, c == 0, &xr, st, c + 1 == p.vcycles_H ? w + 2 : nullptr, 4));
    if (!tiled(L)) {
      ProfScope ps(st, K_VSTORE, sizeof(T) == 4, n * (16.0 + 2.0 * sizeof(T)), 0.0);
      launch_k(L.pdl, k_store2<T, V2>, blocks_for(n), TPB, 0, st, n, xr, w + 2, 4);
    }
    CH_LAUNCHED();
  }
  if (fork) CH_CUDA(cudaStreamWaitEvent(st, pc->ev_join, 0));
  return CH_OK;
}

ch_status precond_apply(ch_precond_s* pc, const double* v, double* w, cudaStream_t st) {
  if (pc->precision == 0)
    return precond_t<double>(pc, pc->hM->Ld, pc->hH->Ld, pc->hM->cinv, pc->hH->cinv, v, w, st);
  return precond_t<float>(pc, pc->hM->Lf, pc->hH->Lf, pc->hM->cinvf, pc->hH->cinvf, v, w, st);
}

// Algorithm 1's step 1 alone on two right-hand sides (N x 2): x = M~^-1 b
template <typename T>
static ch_status mass_solve_t(ch_precond_s* pc, std::vector<LevelT<T>>& LM, const T* cinvM, const double* b,
                              double* x, cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  const ch_params& p = pc->sys->p;
  LevelT<T>& L = LM[0];
  const int n = L.A.nrows;
  k_load2<T, V2><<<blocks_for(n), TPB, 0, st>>>(n, b, 2, L.b);
  CH_LAUNCHED();
  V2* xr = L.x;
  if (p.precond_M == 1) {
    CH_TRY(semi_iteration<T>(L, pc->sys->mesh->dim, semi_steps(p), &xr, st));
  } else {
    for (int c = 0; c < p.vcycles_M; ++c) CH_TRY(vcycle<T>(pc->hM, LM.data(), cinvM, 0, c == 0, &xr, st));
  }
  k_store2<T, V2><<<blocks_for(n), TPB, 0, st>>>(n, xr, x, 2);
  CH_LAUNCHED();
  return CH_OK;
}

ch_status mass_solve(ch_precond_s* pc, const double* b, double* x, cudaStream_t st) {
  if (pc->precision == 0) return mass_solve_t<double>(pc, pc->hM->Ld, pc->hM->cinv, b, x, st);
  return mass_solve_t<float>(pc, pc->hM->Lf, pc->hM->cinvf, b, x, st);
}

}  // namespace ch

// ---------------------------------------------------------------- allocation-free V-cycles
// ch_vcycle_noalloc runs the same V-cycles as ch_vcycle, but the per-level work vectors
// (x, x2, r, b for every level, two right-hand sides each) are carved out of one
// file-scope device array instead of the preconditioner's own buffers, so a call needs no
// device memory beyond the caller's b and x and the already-built hierarchy.  The array is
// reserved in every GPU that loads the library for the life of the process.
namespace ch {

constexpr size_t NOALLOC_SCRATCH_BYTES = size_t(8) << 20;  // 8 MiB per device
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

namespace {
constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// The array's device address for the current device.  In host code the symbol names a host
// stand-in, so the address is looked up once per device (with that device current) and cached.
ch_status noalloc_scratch(void** out) {
  int dev = -1;
  CH_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
    set_error("ch_vcycle_noalloc: device ordinal %d not supported (max %d)", dev, NOALLOC_MAX_DEVICES);
    return CH_ERR_ARG;
  }
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || p == nullptr) {
      set_error("ch_vcycle_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
      return CH_ERR_CUDA;
    }
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return CH_OK;
}
}  // namespace

template <typename T>
static ch_status solve_static(Hierarchy* h, const std::vector<LevelT<T>>& src, const T* cinv,
                              const double* b, double* x, int ncyc, cudaStream_t st) {
  using V2 = typename V2T<T>::t;
  constexpr int MAXLEV = 32;
  if (h->nlev > MAXLEV) {
    set_error("ch_vcycle_noalloc: hierarchy has %d levels (max %d)", h->nlev, MAXLEV);
    return CH_ERR_ARG;
  }
  // The documented limit: 5 vectors of n_l pairs per level, each rounded up to 256 bytes (4 are used)
  size_t need = 0;
  for (int l = 0; l < h->nlev; ++l) need += 5 * ((src[l].A.nrows * sizeof(V2) + 255) / 256 * 256);
  if (need > NOALLOC_SCRATCH_BYTES) {
    set_error("ch_vcycle_noalloc: hierarchy needs %zu bytes of work space, the static array holds %zu "
              "(use ch_vcycle for this size)", need, NOALLOC_SCRATCH_BYTES);
    return CH_ERR_ARG;
  }
  void* base = nullptr;
  CH_TRY(noalloc_scratch(&base));
  LevelT<T> Ls[MAXLEV];
  unsigned char* cur = static_cast<unsigned char*>(base);
  auto carve = [&](int n) {
    V2* p = reinterpret_cast<V2*>(cur);
    cur += (n * sizeof(V2) + 255) / 256 * 256;
    return p;
  };
  for (int l = 0; l < h->nlev; ++l) {
    Ls[l] = src[l];  // matrices, diagonal inverses: the hierarchy's own
    const int n = src[l].A.nrows;
    Ls[l].x = carve(n);
    Ls[l].x2 = carve(n);
    Ls[l].r = carve(n);
    Ls[l].b = carve(n);
  }
  // Every work vector is written before it is read (zero initial guesses are applied by the
  // first Chebyshev step), so nothing in the array needs clearing between calls.
  const int n0 = Ls[0].A.nrows;
  k_load2<T, V2><<<blocks_for(n0), TPB, 0, st>>>(n0, b, 2, Ls[0].b);
  CH_LAUNCHED();
  V2* xr = Ls[0].x;
  for (int c = 0; c < ncyc; ++c) CH_TRY(vcycle<T>(h, Ls, cinv, 0, c == 0, &xr, st));
  k_store2<T, V2><<<blocks_for(n0), TPB, 0, st>>>(n0, xr, x, 2);
  CH_LAUNCHED();
  return CH_OK;
}

ch_status hierarchy_solve_noalloc(Hierarchy* h, const double* b, double* x, int ncyc, cudaStream_t st) {
  if (h->precision == 0) return solve_static<double>(h, h->Ld, h->cinv, b, x, ncyc, st);
  return solve_static<float>(h, h->Lf, h->cinvf, b, x, ncyc, st);
}

}  // namespace ch
