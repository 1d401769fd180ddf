// Mesh generation, P1 assembly, explicit loads and the block operator of Eq. (14).
//
// Everything is node-centric ("gather"): the thread of node i visits the simplices, cells or
// boundary facets incident to i in increasing index order and adds their contributions,
// so every sum has a fixed order and results are bitwise reproducible (no atomics).
#include <algorithm>
#include <cmath>

#include "ch_internal.cuh"

namespace ch {

// ---------------------------------------------------------------- mesh (Section 4)
__global__ void k_fill_int(int* a, int n, int v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = v;
}

__global__ void k_mesh_nodes(ch_params p, int N, int node_off, double* coords) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const int i = n % (p.nx + 1);
  const int j = (n / (p.nx + 1)) % (p.ny + 1);
  const int g = node_off + n;
  if (p.dim == 2) {
    coords[2 * g + 0] = i * (p.Lx / p.nx);
    coords[2 * g + 1] = j * (p.Ly / p.ny);
  } else {
    const int k = n / ((p.nx + 1) * (p.ny + 1));
    coords[3 * g + 0] = i * (p.Lx / p.nx);
    coords[3 * g + 1] = j * (p.Ly / p.ny);
    coords[3 * g + 2] = k * (p.Lz / p.nz);
  }
}

// 2D: cell c = i + nx j -> triangles 2c = (v00, v10, v11), 2c+1 = (v00, v11, v01).
// 3D: hexahedron c -> the 6 Kuhn tetrahedra v000 -> +e_a -> +e_a+e_b -> v111 over the
// permutations (a,b,c) of the axes, in lexicographic order of the permutation.
__global__ void k_mesh_elems(ch_params p, int E, int node_off, int* el) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  if (p.dim == 2) {
    const int c = e >> 1, i = c % p.nx, j = c / p.nx;
    const int v00 = node_off + i + (p.nx + 1) * j, v10 = v00 + 1, v01 = v00 + p.nx + 1, v11 = v01 + 1;
    if ((e & 1) == 0) {
      el[3 * e] = v00; el[3 * e + 1] = v10; el[3 * e + 2] = v11;
    } else {
      el[3 * e] = v00; el[3 * e + 1] = v11; el[3 * e + 2] = v01;
    }
  } else {
    const int c = e / 6, t = e % 6;
    const int i = c % p.nx, j = (c / p.nx) % p.ny, k = c / (p.nx * p.ny);
    const int s[3] = {1, p.nx + 1, (p.nx + 1) * (p.ny + 1)};
    const int perm[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
    const int v0 = node_off + i + s[1] * j + s[2] * k;
    el[4 * e + 0] = v0;
    el[4 * e + 1] = v0 + s[perm[t][0]];
    el[4 * e + 2] = v0 + s[perm[t][0]] + s[perm[t][1]];
    el[4 * e + 3] = v0 + s[0] + s[1] + s[2];
  }
}

// Boundary facets of the Kuhn / diagonal split on y = 0 (bottom) and y = Ly (top).
__global__ void k_mesh_facets(ch_params p, int F, int node_off, int* bot, int* top) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= F) return;
  if (p.dim == 2) {
    const int b = node_off + f, t = node_off + p.ny * (p.nx + 1) + f;
    bot[2 * f] = b; bot[2 * f + 1] = b + 1;
    top[2 * f] = t; top[2 * f + 1] = t + 1;
  } else {
    const int q = f >> 1, i = q % p.nx, k = q / p.nx;
    const int sx = 1, sz = (p.nx + 1) * (p.ny + 1);
    const int b = node_off + i + sz * k;                      // (i, 0, k)
    const int t = node_off + i + (p.nx + 1) * p.ny + sz * k;  // (i, ny, k)
    if ((f & 1) == 0) {
      bot[3 * f] = b; bot[3 * f + 1] = b + sx; bot[3 * f + 2] = b + sx + sz;
      top[3 * f] = t; top[3 * f + 1] = t + sx; top[3 * f + 2] = t + sx + sz;
    } else {
      bot[3 * f] = b; bot[3 * f + 1] = b + sz; bot[3 * f + 2] = b + sx + sz;
      top[3 * f] = t; top[3 * f + 1] = t + sz; top[3 * f + 2] = t + sx + sz;
    }
  }
}

// |T| and barycentric gradients: lambda_{1..d} = J^{-1}(x - x_0), J = [x_1-x_0, ..., x_d-x_0].
template <int D>
__device__ __forceinline__ double simplex_geo(const double* coords, const int* v, double g[D + 1][D]);

template <>
__device__ __forceinline__ double simplex_geo<2>(const double* X, const int* v, double g[3][2]) {
  const double x0 = X[2 * v[0]], y0 = X[2 * v[0] + 1];
  const double j00 = X[2 * v[1]] - x0, j10 = X[2 * v[1] + 1] - y0;
  const double j01 = X[2 * v[2]] - x0, j11 = X[2 * v[2] + 1] - y0;
  const double det = j00 * j11 - j01 * j10;
  const double id = 1.0 / det;
  g[1][0] = j11 * id;  g[1][1] = -j01 * id;
  g[2][0] = -j10 * id; g[2][1] = j00 * id;
  g[0][0] = -(g[1][0] + g[2][0]);
  g[0][1] = -(g[1][1] + g[2][1]);
  return 0.5 * fabs(det);
}

template <>
__device__ __forceinline__ double simplex_geo<3>(const double* X, const int* v, double g[4][3]) {
  double e[3][3];
  for (int a = 0; a < 3; ++a)
    for (int c = 0; c < 3; ++c) e[a][c] = X[3 * v[a + 1] + c] - X[3 * v[0] + c];
  // rows of J^{-1}: (e2 x e3, e3 x e1, e1 x e2) / det
  double r[3][3];
  for (int a = 0; a < 3; ++a) {
    const double* u = e[(a + 1) % 3];
    const double* w = e[(a + 2) % 3];
    r[a][0] = u[1] * w[2] - u[2] * w[1];
    r[a][1] = u[2] * w[0] - u[0] * w[2];
    r[a][2] = u[0] * w[1] - u[1] * w[0];
  }
  const double det = e[0][0] * r[0][0] + e[0][1] * r[0][1] + e[0][2] * r[0][2];
  const double id = 1.0 / det;
  for (int c = 0; c < 3; ++c) {
    g[1][c] = r[0][c] * id;
    g[2][c] = r[1][c] * id;
    g[3][c] = r[2][c] * id;
    g[0][c] = -(g[1][c] + g[2][c] + g[3][c]);
  }
  return fabs(det) / 6.0;
}

template <int D>
__global__ void k_elem_vol(const double* X, const int* el, int E, double* vol) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  double g[D + 1][D];
  vol[e] = simplex_geo<D>(X, el + (D + 1) * e, g);
}

// facet measure: segment length (2D) or triangle area (3D)
template <int D>
__global__ void k_facet_vol(const double* X, const int* f, int F, double* vol) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= F) return;
  if (D == 2) {
    const double dx = X[2 * f[2 * q + 1]] - X[2 * f[2 * q]];
    const double dy = X[2 * f[2 * q + 1] + 1] - X[2 * f[2 * q] + 1];
    vol[q] = sqrt(dx * dx + dy * dy);
  } else {
    double u[3], w[3];
    for (int c = 0; c < 3; ++c) {
      u[c] = X[3 * f[3 * q + 1] + c] - X[3 * f[3 * q] + c];
      w[c] = X[3 * f[3 * q + 2] + c] - X[3 * f[3 * q] + c];
    }
    const double cx = u[1] * w[2] - u[2] * w[1], cy = u[2] * w[0] - u[0] * w[2],
                 cz = u[0] * w[1] - u[1] * w[0];
    vol[q] = 0.5 * sqrt(cx * cx + cy * cy + cz * cz);
  }
}

// class id of every node of one run (Lattice) from the classes along its axes (nx + 1, ny + 1 and in 3D
// nz + 1 of them), ncx and ncy of which are distinct on the first two
__global__ void k_lat_ids(ch_params p, int N, int node_off, const int* axes, int ncx, int ncy, int base, int id32,
                          void* out) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  const int i = n % (p.nx + 1), j = (n / (p.nx + 1)) % (p.ny + 1);
  int c = axes[i] + ncx * axes[p.nx + 1 + j];
  if (p.dim == 3) c += ncx * ncy * axes[p.nx + p.ny + 2 + n / ((p.nx + 1) * (p.ny + 1))];
  if (id32) static_cast<int*>(out)[node_off + n] = base + c;
  else static_cast<uint16_t*>(out)[node_off + n] = (uint16_t)(base + c);
}

// The classes of one axis (appended to cls, one per node) and a node of each: by position, or by the widths
// of the cells on either side, computed as k_mesh_nodes and the element matrices do (volatile: no fused
// multiply-add, the coordinates are rounded; the set-up checks find a difference).
static std::vector<int> axis_classes(int cells, double length, bool widths, std::vector<int>& cls) {
  if (!widths) {
    for (int i = 0; i <= cells; ++i) cls.push_back(i == 0 ? 0 : (i == cells ? 2 : 1));
    return {0, cells / 2, cells};
  }
  std::vector<int> rep;
  std::vector<double> left, right;
  const double h = length / cells;
  double before = 0.0;
  size_t at = 0;
  for (int i = 0; i <= cells; ++i) {
    volatile double x0 = i * h, x1 = (i + 1) * h;
    const double after = i < cells ? x1 - x0 : 0.0;
    const auto is = [&](size_t q) { return left[q] == before && right[q] == after; };
    if (at >= rep.size() || !is(at)) {  // (mostly the class of the node before)
      for (at = 0; at < rep.size() && !is(at); ++at) {}
      if (at == rep.size()) {
        rep.push_back(i);
        left.push_back(before);
        right.push_back(after);
      }
    }
    cls.push_back((int)at);
    before = after;
  }
  return rep;
}

static ch_status lattice_build(ch_mesh_s* m, bool widths, Lattice* L, cudaStream_t st) {
  const int R = (int)m->runs.size(), d = m->dim;
  struct Run {
    size_t axes;
    int ncx, ncy, base;
  };
  std::vector<Run> runs(R);
  std::vector<int> cls, rep;
  std::vector<int2> wh;
  int64_t nids = 0;
  for (int r = 0; r < R; ++r) {
    const ch_params& p = m->runs[r];
    const size_t axes = cls.size();
    const std::vector<int> rx = axis_classes(p.nx, p.Lx, widths, cls), ry = axis_classes(p.ny, p.Ly, widths, cls);
    const std::vector<int> rz = d == 3 ? axis_classes(p.nz, p.Lz, widths, cls) : std::vector<int>{0};
    runs[r] = {axes, (int)rx.size(), (int)ry.size(), (int)nids};
    nids += (int64_t)rx.size() * ry.size() * rz.size();
    if (nids > 2000000000LL) {
      set_error("batched mesh too large for int32 indexing");
      return CH_ERR_ARG;
    }
    const int W = p.nx + 1, WH = W * (p.ny + 1);
    for (int z : rz)
      for (int y : ry)
        for (int x : rx) {
          wh.push_back(make_int2(W, WH));
          rep.push_back(m->run_off[r] + x + W * y + WH * z);
        }
  }
  L->dim = d;
  L->ncls = widths ? 0 : (d == 2 ? 9 : 27);
  L->nids = (int)nids;
  L->multi = R > 1;
  L->W = m->runs[0].nx + 1;
  L->WH = L->W * (m->runs[0].ny + 1);
  L->id32 = L->nids > 65536;
  uint8_t* ids = nullptr;
  int* axes = nullptr;
  CH_TRY(m->mem.get(&ids, (size_t)m->N * (L->id32 ? 4 : 2)));
  CH_TRY(m->mem.get(&axes, cls.size()));
  CH_TRY(m->mem.get(&L->wh, wh.size()));
  CH_TRY(m->mem.get(&L->rep, rep.size()));
  L->id = ids;
  CH_CUDA(cudaMemcpyAsync(axes, cls.data(), sizeof(int) * cls.size(), cudaMemcpyHostToDevice, st));
  CH_CUDA(cudaMemcpyAsync(L->wh, wh.data(), sizeof(int2) * wh.size(), cudaMemcpyHostToDevice, st));
  CH_CUDA(cudaMemcpyAsync(L->rep, rep.data(), sizeof(int) * rep.size(), cudaMemcpyHostToDevice, st));
  for (int r = 0; r < R; ++r) {
    const int n = m->run_off[r + 1] - m->run_off[r];
    k_lat_ids<<<blocks_for(n), TPB, 0, st>>>(m->runs[r], n, m->run_off[r], axes + runs[r].axes, runs[r].ncx,
                                             runs[r].ncy, runs[r].base, L->id32, L->id);
  }
  CH_LAUNCHED();
  CH_CUDA(cudaStreamSynchronize(st));  // the host arrays end here
  return CH_OK;
}

// counts of one box mesh
static void box_counts(const ch_params& p, int* N, int* E, int* F) {
  if (p.dim == 2) {
    *N = (p.nx + 1) * (p.ny + 1);
    *E = 2 * p.nx * p.ny;
    *F = p.nx;
  } else {
    *N = (p.nx + 1) * (p.ny + 1) * (p.nz + 1);
    *E = 6 * p.nx * p.ny * p.nz;
    *F = 2 * p.nx * p.nz;
  }
}

// The mesh of every run, laid out one after another: run r owns nodes [run_off[r], run_off[r+1]),
// its elements and boundary facets follow those of run r-1 and reference only its own nodes, so
// the union is a disjoint set of box meshes (one run: the plain mesh).
ch_status mesh_build(ch_mesh_s* m, cudaStream_t st) {
  const int R = (int)m->runs.size();
  const int d = m->runs[0].dim;
  m->dim = d;
  m->p = m->runs[0];
  m->run_off.assign(R + 1, 0);
  std::vector<int> eoff(R + 1, 0), foff(R + 1, 0);
  for (int r = 0; r < R; ++r) {
    int n, e, f;
    box_counts(m->runs[r], &n, &e, &f);
    if ((int64_t)m->run_off[r] + n > 2000000000LL) {
      set_error("batched mesh too large for int32 indexing");
      return CH_ERR_ARG;
    }
    m->run_off[r + 1] = m->run_off[r] + n;
    eoff[r + 1] = eoff[r] + e;
    foff[r + 1] = foff[r] + f;
  }
  m->N = m->run_off[R];
  m->E = eoff[R];
  m->Fb = m->Ft = foff[R];
  CH_TRY(m->mem.get(&m->coords, (size_t)m->N * d));
  CH_TRY(m->mem.get(&m->elems, (size_t)m->E * (d + 1)));
  CH_TRY(m->mem.get(&m->bot, (size_t)m->Fb * d));
  CH_TRY(m->mem.get(&m->top, (size_t)m->Ft * d));
  CH_TRY(m->mem.get(&m->vol, (size_t)m->E));
  CH_TRY(m->mem.get(&m->bvol, (size_t)m->Fb));
  CH_TRY(m->mem.get(&m->tvol, (size_t)m->Ft));
  CH_TRY(m->mem.get(&m->node_run, (size_t)m->N));
  CH_TRY(m->mem.get(&m->run_off_d, (size_t)R + 1));
  CH_TRY(lattice_build(m, true, &m->lat, st));
  CH_TRY(lattice_build(m, false, &m->pos, st));
  std::vector<CellGrid> grid(R);
  for (int r = 0; r < R; ++r) {
    const ch_params& p = m->runs[r];
    grid[r] = {m->run_off[r], eoff[r] / (d == 2 ? 2 : 6), p.nx, p.ny, d == 3 ? p.nz : 0};
  }
  CH_TRY(m->mem.get(&m->cell_grid, (size_t)R));
  CH_CUDA(cudaMemcpyAsync(m->cell_grid, grid.data(), sizeof(CellGrid) * R, cudaMemcpyHostToDevice, st));
  for (int r = 0; r < R; ++r) {
    const ch_params& p = m->runs[r];
    const int n = m->run_off[r + 1] - m->run_off[r], e = eoff[r + 1] - eoff[r], f = foff[r + 1] - foff[r];
    k_mesh_nodes<<<blocks_for(n), TPB, 0, st>>>(p, n, m->run_off[r], m->coords);
    k_mesh_elems<<<blocks_for(e), TPB, 0, st>>>(p, e, m->run_off[r], m->elems + (size_t)eoff[r] * (d + 1));
    k_mesh_facets<<<blocks_for(f), TPB, 0, st>>>(p, f, m->run_off[r], m->bot + (size_t)foff[r] * d,
                                                  m->top + (size_t)foff[r] * d);
    k_fill_int<<<blocks_for(n), TPB, 0, st>>>(m->node_run + m->run_off[r], n, r);
  }
  CH_LAUNCHED();
  CH_CUDA(cudaMemcpyAsync(m->run_off_d, m->run_off.data(), sizeof(int) * (R + 1), cudaMemcpyHostToDevice, st));
  if (d == 2) {
    k_elem_vol<2><<<blocks_for(m->E), TPB, 0, st>>>(m->coords, m->elems, m->E, m->vol);
    k_facet_vol<2><<<blocks_for(m->Fb), TPB, 0, st>>>(m->coords, m->bot, m->Fb, m->bvol);
    k_facet_vol<2><<<blocks_for(m->Ft), TPB, 0, st>>>(m->coords, m->top, m->Ft, m->tvol);
  } else {
    k_elem_vol<3><<<blocks_for(m->E), TPB, 0, st>>>(m->coords, m->elems, m->E, m->vol);
    k_facet_vol<3><<<blocks_for(m->Fb), TPB, 0, st>>>(m->coords, m->bot, m->Fb, m->bvol);
    k_facet_vol<3><<<blocks_for(m->Ft), TPB, 0, st>>>(m->coords, m->top, m->Ft, m->tvol);
  }
  CH_LAUNCHED();
  CH_TRY(build_incidence(m->elems, m->E, d + 1, m->N, &m->n2e_ptr, &m->n2e, st, m->mem));
  CH_TRY(build_incidence(m->bot, m->Fb, d, m->N, &m->n2b_ptr, &m->n2b, st, m->mem));
  CH_TRY(build_incidence(m->top, m->Ft, d, m->N, &m->n2t_ptr, &m->n2t, st, m->mem));
  return CH_OK;
}

// ---------------------------------------------------------------- CSR pattern
constexpr int MAXADJ = 128;  // distinct-or-not vertex entries gathered per node

__device__ int gather_adjacent(const int* el, int k, const int* ptr, const int* list, int v,
                               int* buf, int* overflow) {
  int n = 0;
  for (int q = ptr[v]; q < ptr[v + 1]; ++q) {
    const int e = list[q];
    for (int a = 0; a < k; ++a) {
      if (n < MAXADJ) buf[n++] = el[k * e + a];
      else *overflow = 1;
    }
  }
  // insertion sort + unique
  for (int i = 1; i < n; ++i) {
    const int x = buf[i];
    int j = i - 1;
    while (j >= 0 && buf[j] > x) {
      buf[j + 1] = buf[j];
      --j;
    }
    buf[j + 1] = x;
  }
  int u = 0;
  for (int i = 0; i < n; ++i)
    if (u == 0 || buf[u - 1] != buf[i]) buf[u++] = buf[i];
  return u;
}

__global__ void k_pattern(const int* el, int k, const int* ptr, const int* list, int N,
                          const int* rowptr, int* cnt, int* col, int* overflow) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= N) return;
  int buf[MAXADJ];
  const int u = gather_adjacent(el, k, ptr, list, v, buf, overflow);
  if (rowptr == nullptr) {
    cnt[v] = u;
  } else {
    for (int i = 0; i < u; ++i) col[rowptr[v] + i] = buf[i];
  }
}

// ---------------------------------------------------------------- values of M and K
__device__ __forceinline__ int find_col(const int* col, int b, int e, int c) {
  while (b < e) {  // binary search in a sorted row
    const int m = (b + e) >> 1;
    if (col[m] < c) b = m + 1;
    else e = m;
  }
  return b;
}

template <int D>
__global__ void k_assemble(const double* X, const int* el, const int* ptr, const int* list, int N,
                           const int* rowptr, const int* col, double* valM, double* valK,
                           int* diag) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= N) return;
  const int rb = rowptr[v], re = rowptr[v + 1];
  for (int q = rb; q < re; ++q) {
    valM[q] = 0.0;
    valK[q] = 0.0;
  }
  diag[v] = find_col(col, rb, re, v);
  constexpr double mscale = 1.0 / ((D + 1) * (D + 2));  // M_e = |T| (1 + delta_ab) / ((d+1)(d+2))
  for (int q = ptr[v]; q < ptr[v + 1]; ++q) {
    const int e = list[q];
    const int* ev = el + (D + 1) * e;
    double g[D + 1][D];
    const double vol = simplex_geo<D>(X, ev, g);
    int a = 0;
    while (ev[a] != v) ++a;
    for (int b = 0; b <= D; ++b) {
      double kab = 0.0;
      for (int c = 0; c < D; ++c) kab = fma(g[a][c], g[b][c], kab);
      const int pos = find_col(col, rb, re, ev[b]);
      if (pos < re && col[pos] == ev[b]) {  // always true: the row pattern holds every neighbour
        valK[pos] += vol * kab;
        valM[pos] += vol * mscale * (a == b ? 2.0 : 1.0);
      }
    }
  }
}

__global__ void k_axpby_vals(const double* x, const double* y, double a, double b, double* z,
                             int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) z[i] = a * x[i] + b * y[i];
}

// ---------------------------------------------------------------- patterned substrate (Section 4)
// With pattern = 1 the substrate energy density of Eq. (5) carries p_p(x) = 1 on the 1st, 3rd and
// 5th sixth of [0, Lx] and p_nfa(x) = 1 on the others (0 elsewhere).  Its boundary load needs, per
// bottom facet F and species s, W1_i = int_F p_s lambda_i and W2_ai = int_F p_s lambda_a lambda_i.
// p_s is constant between breakpoints, so F is clipped to each sixth [lo, hi] and the pieces are
// integrated exactly with the vertex-value rules for linear u, v on a simplex S of dimension k:
//   int_S u = |S| / (k+1) sum_j u_j,   int_S u v = |S| / ((k+1)(k+2)) (sum_j u_j v_j + sum u sum v).
// A 3D facet (a triangle in the x-z plane y = 0) is clipped by Sutherland-Hodgman against the two
// half-planes and fanned into triangles; a 2D facet is a segment of the x axis.
template <int D>
struct FacetHat {  // the facet's hat functions as affine functions of (x, z)
  double X[D], Z[D], det;
  __device__ void lam(double x, double z, double* l) const {
    if constexpr (D == 2) {
      l[1] = (x - X[0]) / (X[1] - X[0]);
      l[0] = 1.0 - l[1];
    } else {
      const double dx = x - X[0], dz = z - Z[0];
      l[1] = (dx * (Z[2] - Z[0]) - (X[2] - X[0]) * dz) / det;
      l[2] = ((X[1] - X[0]) * dz - dx * (Z[1] - Z[0])) / det;
      l[0] = 1.0 - l[1] - l[2];
    }
  }
};

// Adds the integrals over the simplex with vertices P (k + 1 = D of them, measure meas) to W.
template <int D>
__device__ void add_piece(const FacetHat<D>& F, const double (*P)[2], double meas, double* W1, double* W2) {
  double L[D][D];  // L[j][i] = lambda_i at vertex j of the piece
#pragma unroll
  for (int j = 0; j < D; ++j) F.lam(P[j][0], P[j][1], L[j]);
  const double c1 = meas / D, c2 = meas / (D * (D + 1));
#pragma unroll
  for (int i = 0; i < D; ++i) {
    double si = 0.0;
#pragma unroll
    for (int j = 0; j < D; ++j) si += L[j][i];
    W1[i] += c1 * si;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      double sa = 0.0, sai = 0.0;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        sa += L[j][a];
        sai += L[j][a] * L[j][i];
      }
      W2[a * D + i] += c2 * (sai + sa * si);
    }
  }
}

// Clips the convex polygon (x, z)[n] to the half-plane sgn (x - c) >= 0; returns the new vertex
// count.  Each clip adds at most one vertex (a triangle ends with at most 5); cap bounds the
// output all the same.
__device__ int clip_x(const double (*in)[2], int n, double c, double sgn, double (*out)[2], int cap) {
  int k = 0;
  for (int j = 0; j < n && k + 2 <= cap; ++j) {
    const double* P = in[j];
    const double* Q = in[(j + 1) % n];
    const double dp = sgn * (P[0] - c), dq = sgn * (Q[0] - c);
    if (dp >= 0.0) {
      out[k][0] = P[0];
      out[k][1] = P[1];
      ++k;
    }
    if ((dp >= 0.0) != (dq >= 0.0)) {
      const double t = dp / (dp - dq);
      out[k][0] = c;
      out[k][1] = P[1] + t * (Q[1] - P[1]);
      ++k;
    }
  }
  return k;
}

template <int D>
__global__ void k_facet_pattern(const double* coords, const int* bot, int nf, double Lx, double* bw) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nf) return;
  constexpr int NW = D + D * D;
  const int* fv = bot + D * f;
  FacetHat<D> F;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    F.X[a] = coords[(size_t)D * fv[a]];
    F.Z[a] = (D == 3) ? coords[(size_t)D * fv[a] + 2] : 0.0;
  }
  F.det = 0.0;
  if constexpr (D == 3) F.det = (F.X[1] - F.X[0]) * (F.Z[2] - F.Z[0]) - (F.X[2] - F.X[0]) * (F.Z[1] - F.Z[0]);
  double W[2][NW];
#pragma unroll
  for (int q = 0; q < 2 * NW; ++q) W[q / NW][q % NW] = 0.0;
  for (int k = 0; k < 6; ++k) {
    const double lo = k * (Lx / 6.0), hi = (k + 1) * (Lx / 6.0);
    double* W1 = W[k & 1];  // species 0 (polymer) on k = 0, 2, 4; species 1 (NFA) on k = 1, 3, 5
    double* W2 = W1 + D;
    if constexpr (D == 2) {
      const double xa = fmax(fmin(F.X[0], F.X[1]), lo), xb = fmin(fmax(F.X[0], F.X[1]), hi);
      if (xb <= xa) continue;
      const double P[2][2] = {{xa, 0.0}, {xb, 0.0}};
      add_piece<D>(F, P, xb - xa, W1, W2);
    } else {
      double A[8][2], B[8][2];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        A[a][0] = F.X[a];
        A[a][1] = F.Z[a];
      }
      int n = clip_x(A, 3, lo, 1.0, B, 8);
      n = clip_x(B, n, hi, -1.0, A, 8);
      for (int j = 1; j + 1 < n; ++j) {
        const double P[3][2] = {{A[0][0], A[0][1]}, {A[j][0], A[j][1]}, {A[j + 1][0], A[j + 1][1]}};
        const double meas = 0.5 * fabs((P[1][0] - P[0][0]) * (P[2][1] - P[0][1]) -
                                       (P[2][0] - P[0][0]) * (P[1][1] - P[0][1]));
        if (meas > 0.0) add_piece<D>(F, P, meas, W1, W2);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 2 * NW; ++q) bw[(size_t)f * 2 * NW + q] = W[q / NW][q % NW];
}

static ch_status log_tables(ch_system_s* s, cudaStream_t st);

// Weights of every run's bottom facets (each run's box is [0, Lx_r] in x).
static ch_status substrate_weights(const ch_mesh_s* m, ch_system_s* s, cudaStream_t st) {
  const int d = m->dim, R = (int)m->runs.size();
  CH_TRY(s->mem.get(&s->bw, (size_t)m->Fb * 2 * (d + d * d)));
  int f0 = 0;
  for (int r = 0; r < R; ++r) {
    int n, e, f;
    box_counts(m->runs[r], &n, &e, &f);
    const int* bot = m->bot + (size_t)f0 * d;
    double* bw = s->bw + (size_t)f0 * 2 * (d + d * d);
    if (f > 0) {
      if (d == 2)
        k_facet_pattern<2><<<blocks_for(f), TPB, 0, st>>>(m->coords, bot, f, m->runs[r].Lx, bw);
      else
        k_facet_pattern<3><<<blocks_for(f), TPB, 0, st>>>(m->coords, bot, f, m->runs[r].Lx, bw);
    }
    f0 += f;
  }
  CH_LAUNCHED();
  return CH_OK;
}

// ---------------------------------------------------------------- the operator's lattice table
template <int ND>
__global__ void k_lat_operator(int nids, const int* rep, const int2* wh, const int* rowptr, const int* col,
                               const double* valM, const double* valK, double* tab) {
  using X = LatAxes<ND>;
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= nids) return;
  const int i = rep[id];
  const int2 w = wh[id];
  double* t = tab + (size_t)id * X::TS;
  for (int k = 0; k < X::TS; ++k) t[k] = 0.0;
  for (int q = rowptr[i]; q < rowptr[i + 1]; ++q)
    for (int d = 0; d < ND; ++d)
      if (lat_off(ND, d, w.x, w.y) == col[q] - i) {
        t[d] = valM[q];
        if (X::index(d) >= 0) t[ND + X::index(d)] = valK[q];
      }
}

// bad = 1 where a row is not its class's table row bit for bit, apart from K's entries off the axes: zero but
// for the rounding of the products in the tetrahedra's gradients (2^-50 of the diagonal at most)
template <int ND>
__global__ void k_lat_operator_check(Lattice L, int N, const int* rowptr, const int* col, const double* valM,
                                     const double* valK, const double* tab, int* bad) {
  using X = LatAxes<ND>;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const int id = lat_id(L, i);
  const int2 w = L.wh[id];
  const double* t = tab + (size_t)id * X::TS;
  const double tk = 0x1p-50 * fabs(t[ND + X::index(ND / 2)]);
  bool ok = true;
  unsigned seen = 0;
  for (int q = rowptr[i]; q < rowptr[i + 1]; ++q) {
    int at = -1;
    for (int d = 0; d < ND; ++d)
      if (lat_off(ND, d, w.x, w.y) == col[q] - i) at = d;
    if (at < 0) {
      ok = false;
      continue;
    }
    int e = -1;
    for (int d = 0; d < ND; ++d)
      if (d == at) e = X::index(d);
    // (an entry whose upper word is zero would pass for an absent neighbour)
    if (!(valM[q] == t[at]) || __double2hiint(t[at]) == 0) ok = false;
    if (e >= 0 ? !(valK[q] == t[ND + e]) : !(fabs(valK[q]) <= tk)) ok = false;
    seen |= 1u << at;
  }
  for (int d = 0; d < ND; ++d)
    if (!(seen >> d & 1) && t[d] != 0.0) ok = false;  // the class has an entry that the row lacks
  if (!ok) *bad = 1;
}

static ch_status lattice_operator(const ch_mesh_s* m, ch_system_s* s, int* bad, cudaStream_t st) {
  const Lattice& L = m->lat;
  const int ts = m->dim == 2 ? LatAxes<7>::TS : LatAxes<15>::TS;
  double* tab = nullptr;
  CH_TRY(s->mem.get(&tab, (size_t)L.nids * ts));
  s->lat.L = L;
  s->lat.a = s->a;
  s->lat.c = s->c;
  s->lat.tab = tab;
  if (m->dim == 2) {
    k_lat_operator<7><<<blocks_for(L.nids, 64), 64, 0, st>>>(L.nids, L.rep, L.wh, s->rowptr, s->col, s->valM, s->valK,
                                                             tab);
    k_lat_operator_check<7><<<blocks_for(s->N), TPB, 0, st>>>(L, s->N, s->rowptr, s->col, s->valM, s->valK, tab, bad);
  } else {
    k_lat_operator<15><<<blocks_for(L.nids, 64), 64, 0, st>>>(L.nids, L.rep, L.wh, s->rowptr, s->col, s->valM,
                                                              s->valK, tab);
    k_lat_operator_check<15><<<blocks_for(s->N), TPB, 0, st>>>(L, s->N, s->rowptr, s->col, s->valM, s->valK, tab, bad);
  }
  CH_LAUNCHED();
  return CH_OK;
}

ch_status assemble_system(const ch_mesh_s* m, ch_system_s* s, cudaStream_t st) {
  const int N = m->N, d = m->dim;
  s->N = N;
  Alloc tmp;
  int *cnt = nullptr, *overflow = nullptr;
  CH_TRY(tmp.get(&cnt, (size_t)N));
  CH_TRY(tmp.get(&overflow, 2));  // ... and the lattice operator's misfit flag
  CH_CUDA(cudaMemsetAsync(overflow, 0, 2 * sizeof(int), st));
  k_pattern<<<blocks_for(N), TPB, 0, st>>>(m->elems, d + 1, m->n2e_ptr, m->n2e, N, nullptr, cnt,
                                            nullptr, overflow);
  CH_LAUNCHED();
  CH_TRY(s->mem.get(&s->rowptr, (size_t)N + 1));
  int64_t nnz = 0;
  CH_TRY(scan_i32_to_rowptr(cnt, s->rowptr, N, &nnz, st, tmp));
  s->nnz = nnz;
  CH_TRY(s->mem.get(&s->col, (size_t)nnz));
  CH_TRY(s->mem.get(&s->valM, (size_t)nnz));
  CH_TRY(s->mem.get(&s->valK, (size_t)nnz));
  CH_TRY(s->mem.get(&s->valH, (size_t)nnz));
  CH_TRY(s->mem.get(&s->eload, (size_t)(m->E / (d == 2 ? 2 : 6)) * (d == 2 ? 4 : 8)));
  CH_TRY(s->mem.get(&s->diag, (size_t)N));
  k_pattern<<<blocks_for(N), TPB, 0, st>>>(m->elems, d + 1, m->n2e_ptr, m->n2e, N, s->rowptr,
                                            nullptr, s->col, overflow);
  CH_LAUNCHED();
  if (d == 2)
    k_assemble<2><<<blocks_for(N), TPB, 0, st>>>(m->coords, m->elems, m->n2e_ptr, m->n2e, N,
                                                  s->rowptr, s->col, s->valM, s->valK, s->diag);
  else
    k_assemble<3><<<blocks_for(N), TPB, 0, st>>>(m->coords, m->elems, m->n2e_ptr, m->n2e, N,
                                                  s->rowptr, s->col, s->valM, s->valK, s->diag);
  CH_LAUNCHED();
  // H = a K + sqrt(c) M  (Section 3, matching Schur approximation)
  k_axpby_vals<<<blocks_for(nnz), TPB, 0, st>>>(s->valK, s->valM, s->a, sqrt(s->c), s->valH, nnz);
  CH_LAUNCHED();
  if (s->p.potential == 3) CH_TRY(log_tables(s, st));
  if (s->p.pattern && s->p.bc_mode) CH_TRY(substrate_weights(m, s, st));
  CH_TRY(lattice_operator(m, s, overflow + 1, st));
  int ovf[2] = {0, 0};
  CH_CUDA(cudaMemcpyAsync(ovf, overflow, sizeof(ovf), cudaMemcpyDeviceToHost, st));
  CH_CUDA(cudaStreamSynchronize(st));
  if (ovf[1]) s->lat.tab = nullptr;
  if (ovf[0]) {
    set_error("a node has more than %d incident simplex vertices", MAXADJ);
    return CH_ERR_INTERNAL;
  }
  return CH_OK;
}

// ---------------------------------------------------------------- explicit loads
// Exact integrals of products of linear functions over a simplex T of dimension d:
//   int_T l_1 ... l_n = d! |T| / (d+n)! * sum over permutations pi of {1..n} of
//                       prod over the cycles C of pi of sum_vertices prod_{k in C} l_k(v),
// which follows from int lambda^alpha = d! alpha! |T| / (d+|alpha|)! because alpha! counts
// the permutations fixing an index tuple.  With l = (p, q, q, lambda_i) it gives
//   int p q^2 lambda_i = d!|T|/(d+4)! [ <p><q>^2 + 2<pq><q> + <q^2><p> + 2<pq^2>
//        + p_i(<q>^2 + <q^2>) + 2 q_i(<p><q> + <pq>) + 4 p_i q_i <q> + 2 q_i^2 <p> + 6 p_i q_i^2 ],
// and with (a, b, lambda_i) on a facet of dimension d-1
//   int a b lambda_i = (d-1)!|F|/(d+2)! [ <a><b> + <ab> + a_i<b> + b_i<a> + 2 a_i b_i ],
// where <x> is the sum of x over the simplex's vertices.

struct MeshPod {
  int dim, N, C;                // nodes, cells (the 2 triangles or 6 tetrahedra of a grid cell)
  const int* elems;
  const int* bot;
  const int* top;
  const double* vol;
  const double* bvol;
  const double* tvol;
  const int *n2b_ptr, *n2b, *n2t_ptr, *n2t;
  const int* node_run;
  const CellGrid* grid;         // per run
};

static MeshPod mesh_pod(const ch_mesh_s* s) {
  MeshPod v;
  v.dim = s->dim;
  v.N = s->N;
  v.C = s->E / (s->dim == 2 ? 2 : 6);
  v.elems = s->elems;
  v.bot = s->bot;
  v.top = s->top;
  v.vol = s->vol;
  v.bvol = s->bvol;
  v.tvol = s->tvol;
  v.n2b_ptr = s->n2b_ptr;
  v.n2b = s->n2b;
  v.n2t_ptr = s->n2t_ptr;
  v.n2t = s->n2t;
  v.node_run = s->node_run;
  v.grid = s->cell_grid;
  return v;
}

// Corners of a cell: bit 0 is +x, bit 1 +y, bit 2 +z.  Simplex t of the cell runs from corner 0 over
// path[t][0] (and path[t][1]) to the opposite corner (k_mesh_elems' order of triangles and tetrahedra).
template <int D> struct CellSimplices;
template <> struct CellSimplices<2> {
  static constexpr int NT = 2, NC = 4;
  __host__ __device__ static constexpr int corner(int t, int a) {  // t = 0: (0, 1, 3), 1: (0, 3, 2)
    constexpr int c[2][3] = {{0, 1, 3}, {0, 3, 2}};
    return c[t][a];
  }
};
template <> struct CellSimplices<3> {
  static constexpr int NT = 6, NC = 8;
  __host__ __device__ static constexpr int corner(int t, int a) {
    constexpr int c[6][4] = {{0, 1, 3, 7}, {0, 1, 5, 7}, {0, 2, 3, 7}, {0, 2, 6, 7}, {0, 4, 5, 7}, {0, 4, 6, 7}};
    return c[t][a];
  }
};
// the nodes of a cell's corners, read from its simplices
template <int D>
__device__ __forceinline__ void cell_nodes(const int* elems, int cell, int (&v)[CellSimplices<D>::NC]) {
  using S = CellSimplices<D>;
  const int* e = elems + (size_t)cell * S::NT * (D + 1);
#pragma unroll
  for (int t = 0; t < S::NT; ++t)
#pragma unroll
    for (int a = 0; a <= D; ++a) {
      bool first = true;  // each corner once
#pragma unroll
      for (int q = 0; q < t * (D + 1) + a; ++q)
        if (S::corner(q / (D + 1), q % (D + 1)) == S::corner(t, a)) first = false;
      if (first) v[S::corner(t, a)] = e[t * (D + 1) + a];
    }
}

// eload of the CB cells from c0 on: per corner the simplices' values (part[simplex][vertex][cell]) in simplex order
template <int D, int CB>
__device__ __forceinline__ void cell_sums(const double2 (*part)[D + 1][CB], int c0, int C, double2* __restrict__ eload) {
  using S = CellSimplices<D>;
  for (int e = threadIdx.x; e < CB * S::NC; e += blockDim.x) {
    const int cl = e / S::NC, corner = e % S::NC;
    if (c0 + cl >= C) continue;
    double fp = 0.0, fn = 0.0;
#pragma unroll
    for (int q = 0; q < S::NT; ++q)
#pragma unroll
      for (int a = 0; a <= D; ++a)
        if (S::corner(q, a) == corner) {
          const double2 v = part[q][a][cl];
          fp += v.x;
          fn += v.y;
        }
    eload[((size_t)c0 + cl) * S::NC + corner] = make_double2(fp, fn);
  }
}

struct LoadCoef {
  double cs;      // coefficient of phi_s in f' (0.2 for Eq. (15), 0 otherwise) / ((d+1)(d+2))
  double cubic;   // 7 for Eq. (15), 0 for f' = 0, times d!/(d+4)!
  int bc;         // boundary loads on/off
  double gp, gn, hp, hn, kev;
  const double* bw;  // patterned substrate weights (Fb x 2 x (D + D^2)), or null for p = 1
};

// The loads are formed per grid cell, one entry per corner, and each node then adds its 4 (8) cells'
// entries: eload[(cell NC + corner) 2 + {0, 1}] = int over the cell of f_p' and f_n' against the corner's
// hat function.  Per simplex T with vertex sums <.> the closed form above is, with c = |T| 7 d!/(d+4)!
// and b = |T| 0.2 / ((d+1)(d+2)),
//   c (<p><q>^2 + 2<pq><q> + <q^2><p> + 2<pq^2>) - b (<phi_s> + 1)            element constants
//   + p_i (c (<q>^2 + <q^2>) + b + q_i (4 c <q> + 6 c q_i)) + q_i (2 c (<p><q> + <pq>) + b + 2 c <p> q_i)
// five FMAs per vertex and species.  FP64-pipe bound (about 95 instructions per tetrahedron): 518 us on
// 128 x 128 x 32 cells and 83 us on 512 x 512, where one thread per simplex with a store per vertex
// took 875 and 122 us.  A
// thread takes a cell, so the products of the nodal values are formed once for its simplices and
// there is one entry per corner instead of one per simplex and vertex (a third of the stores in 3D).
template <int D, typename F>
__device__ __forceinline__ void simplex_loads(const double (&P)[D + 1], const double (&Q)[D + 1],
                                              const double (&PQ)[D + 1], double c, double b, F add) {
  const double c_2 = 2.0 * c, c_4 = 4.0 * c, c_6 = 6.0 * c;
  double Sp = 0, Sq = 0, Spq = 0, Spp = 0, Sqq = 0, Spqq = 0, Sppq = 0;
#pragma unroll
  for (int a = 0; a <= D; ++a) {
    Sp += P[a];
    Sq += Q[a];
    Spq += PQ[a];
    Spp = fma(P[a], P[a], Spp);
    Sqq = fma(Q[a], Q[a], Sqq);
    Spqq = fma(PQ[a], Q[a], Spqq);
    Sppq = fma(PQ[a], P[a], Sppq);
  }
  const double bs = b * ((D + 2) - Sp - Sq);  // b (<phi_s> + 1)
  const double cSp = c * Sp, cSq = c * Sq, cpq = c_2 * Spq;
  const double Ap = fma(c_2, Spqq, fma(cSp, fma(Sq, Sq, Sqq), cpq * Sq)) - bs;
  const double An = fma(c_2, Sppq, fma(cSq, fma(Sp, Sp, Spp), cpq * Sp)) - bs;
  const double Bp = fma(c, fma(Sq, Sq, Sqq), b), Bn = fma(c, fma(Sp, Sp, Spp), b);
  const double C = fma(2.0 * cSp, Sq, cpq) + b;
  const double Sp2 = 2.0 * cSp, Sq2 = 2.0 * cSq, Sp4 = c_4 * Sp, Sq4 = c_4 * Sq;
#pragma unroll
  for (int a = 0; a <= D; ++a) {
    const double p = P[a], q = Q[a];
    add(a, fma(p, fma(q, fma(c_6, q, Sq4), Bp), fma(q, fma(Sp2, q, C), Ap)),
        fma(q, fma(p, fma(c_6, p, Sp4), Bn), fma(p, fma(Sq2, p, C), An)));
  }
}

template <int D>
__global__ void __launch_bounds__(128) k_cell_loads(const MeshPod m, LoadCoef L, const double* pp, const double* pn,
                                                    int ld, double2* __restrict__ eload) {
  using S = CellSimplices<D>;
  const int cell = blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= m.C) return;
  int v[S::NC];
  cell_nodes<D>(m.elems, cell, v);
  double P[S::NC], Q[S::NC], PQ[S::NC], Fp[S::NC], Fn[S::NC];
#pragma unroll
  for (int a = 0; a < S::NC; ++a) {
    P[a] = pp[(size_t)ld * v[a]];
    Q[a] = pn[(size_t)ld * v[a]];
    PQ[a] = P[a] * Q[a];
    Fp[a] = Fn[a] = 0.0;
  }
  const double vol = m.vol[(size_t)cell * S::NT];  // the cell's simplices are congruent
  const double c = vol * L.cubic, b = vol * L.cs;  // (common to the cell's nodes, as their roundings are)
#pragma unroll
  for (int t = 0; t < S::NT; ++t) {
    double p[D + 1], q[D + 1], pq[D + 1];
#pragma unroll
    for (int a = 0; a <= D; ++a) {
      p[a] = P[S::corner(t, a)];
      q[a] = Q[S::corner(t, a)];
      pq[a] = PQ[S::corner(t, a)];
    }
    simplex_loads<D>(p, q, pq, c, b, [&](int a, double fp, double fn) {
      Fp[S::corner(t, a)] += fp;
      Fn[S::corner(t, a)] += fn;
    });
  }
#pragma unroll
  for (int a = 0; a < S::NC; ++a) eload[(size_t)cell * S::NC + a] = make_double2(Fp[a], Fn[a]);
}

// The same for meshes of few cells, a thread per simplex (32 cells and a warp per simplex of theirs in a block), whose
// corner values are added in shared memory in simplex order: k_cell_loads' sums, bit for bit.  A warp's FP64
// instructions hold its quarter of the SM 64 clocks each, so six tetrahedra one after another take 20 us however few
// the cells: right-hand sides of 16 x 16 x 16 cells 33 us, 43 by cells.
template <int D>
__global__ void __launch_bounds__(32 * CellSimplices<D>::NT) k_cell_loads_split(const MeshPod m, LoadCoef L,
                                                                                const double* pp, const double* pn,
                                                                                int ld, double2* __restrict__ eload) {
  using S = CellSimplices<D>;
  __shared__ double2 part[S::NT][D + 1][32];
  const int t = threadIdx.x >> 5, in = threadIdx.x & 31, cell0 = blockIdx.x * 32;
  if (cell0 + in < m.C) {
    const int* ev = m.elems + ((size_t)(cell0 + in) * S::NT + t) * (D + 1);
    double P[D + 1], Q[D + 1], PQ[D + 1];
#pragma unroll
    for (int a = 0; a <= D; ++a) {
      P[a] = pp[(size_t)ld * ev[a]];
      Q[a] = pn[(size_t)ld * ev[a]];
      PQ[a] = P[a] * Q[a];
    }
    const double vol = m.vol[(size_t)(cell0 + in) * S::NT];
    simplex_loads<D>(P, Q, PQ, vol * L.cubic, vol * L.cs,
                     [&](int a, double fp, double fn) { part[t][a][in] = make_double2(fp, fn); });
  }
  __syncthreads();
  cell_sums<D, 32>(part, cell0, m.C, eload);
}

// ---- The Flory-Huggins load (potential = 3).  Section 2's bulk energy
//   f = phi_p ln(phi_p) / N_p + phi_n ln(phi_n) / N_n + phi_s ln(phi_s) / N_s
//       + chi_pn phi_p phi_n + chi_ps phi_p phi_s + chi_ns phi_n phi_s,   phi_s = 1 - phi_p - phi_n,
// differentiated through phi_s like Eq. (15):
//   f_p' = (ln phi_p + 1) / N_p - (ln phi_s + 1) / N_s + chi_pn phi_n + chi_ps (phi_s - phi_p) - chi_ns phi_n
//   f_n' = (ln phi_n + 1) / N_n - (ln phi_s + 1) / N_s + (chi_pn - chi_ps) phi_p + chi_ns (phi_s - phi_n)
// with each logarithm taken at max(phi, delta) (a NaN stays a NaN).  The integrand is not a
// polynomial, so a fixed rule defines the load: on every simplex the product of 3-point
// Gauss-Legendre rules collapsed onto it (Duffy), 9 points on a triangle, 27 on a tetrahedron.
// f_p' = ln+ phi_p / N_p - ln+ phi_s / N_s + chi_ps + mix phi_n - 2 chi_ps phi_p and f_n' alike, ln+ x =
// 1 + ln x, mix = chi_pn - chi_ps - chi_ns (mix_lo: what its rounding left out)
struct FhCoef {
  double chi_ps, chi_ns, mix, mix_lo, inv_np, inv_nn, inv_ns, delta;
};
static FhCoef fh_coef(const ch_params& p) {
  const auto rest = [](double a, double b, double d) {  // a - b - d for d = fl(a - b)
    const double t = a - d;
    return (a - (d + t)) + (t - b);
  };
  const double d = p.chi_pn - p.chi_ps, mix = d - p.chi_ns;
  return {p.chi_ps, p.chi_ns, mix, rest(p.chi_pn, p.chi_ps, d) + rest(d, p.chi_ns, mix), 1.0 / p.N_p, 1.0 / p.N_nfa,
          1.0 / p.N_s, p.fh_delta};
}

// Constants and tables are formed in double-double arithmetic (Dekker 1971) and rounded once.
struct DD {
  double h, l;
};
constexpr DD dd_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
constexpr DD dd_prod(double a, double b) {  // exact: products of halves
  const double ca = 134217729.0 * a, ah = ca - (ca - a), al = a - ah;
  const double cb = 134217729.0 * b, bh = cb - (cb - b), bl = b - bh, p = a * b;
  return {p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr DD operator+(DD a, DD b) {
  const DD s = dd_sum(a.h, b.h);
  return dd_sum(s.h, s.l + a.l + b.l);
}
constexpr DD operator*(DD a, DD b) {
  const DD p = dd_prod(a.h, b.h);
  return dd_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr DD dd_div(DD a, DD b) {
  const double q = a.h / b.h;
  const DD p = b * DD{q, 0.0};
  return dd_sum(q, ((a.h - p.h) + (a.l - p.l)) / b.h);
}

// Gauss-Legendre on [0, 1] with 3 points: 1/2 -+ sqrt(15)/10 and 1/2, weights 5/18, 4/9, 5/18.
// Square (u, v) -> triangle (u, v (1 - u)), Jacobian 1 - u; cube (u, v, t) -> tetrahedron
// (u, v (1 - u), t (1 - u)(1 - v)), Jacobian (1 - u)^2 (1 - v); normalised by the reference
// simplex's measure (1/2, 1/6).  The vertices' weights are multiples of 2^-53, so that a point's sum to one
// exactly: a sum off by one rounding is common to all points, and 1 - phi_p - phi_n moves by as much.
constexpr double gl_grid(double x) { return (x + 1.0) - 1.0; }
constexpr DD gl_w(int i) { return dd_div({i == 1 ? 4.0 : 2.5, 0.0}, {9.0, 0.0}); }

// 1 + ln x of a positive value by tables over the mantissa and the exponent (Tang 1990, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic", with his leading and trailing
// parts): x = 2^k m, f the reciprocal of the middle of m's interval (2048 of them) cut to 21 bits, r = m f - 1
// (one FMA, |r| <= 2^-11), 1 + ln x = (k ln 2)_lead + (1 - ln f)_lead + r - r^2 / 2 + t, t = r^3 / 3 - r^4 / 4 +
// r^5 / 5 + (k ln 2)_trail - (ln f)_trail.  The leading parts are multiples of 2^-42, so their sum is exact;
// t, below 2^-34, takes FP32.  Five FP64 instructions (the pipe that bounds the kernel), the rest integer and
// FP32 ones.  Error against extended precision 0.29 ulp of ln x rms and 0.502 at most over [1e-10, 1/2], as a
// correctly rounded logarithm; around x = 1, where f is 1 and 1/2, below 2^-60.  Other values (zero, negative,
// denormal, above 2^65, infinite, NaN) take CUDA's log.
constexpr int LOG_M = 2048, LOG_K = 1088;
struct LogTables {
  double y[LOG_M];  // 1 - ln f, leading part
  double k[LOG_K];  // (biased exponent - 1023) ln 2, leading part
  int f[LOG_M];     // upper word of f, the lower one is zero
  float yt[LOG_M];  // trailing parts
  float kt[LOG_K];
};
static_assert(sizeof(LogTables) % 16 == 0, "copied in 16-byte pieces");
// the same on the device (no contraction into other fused multiply-adds)
__device__ DD dv_sum(double a, double b) {
  const double s = __dadd_rn(a, b), t = __dadd_rn(s, -a);
  return {s, __dadd_rn(__dadd_rn(a, -__dadd_rn(s, -t)), __dadd_rn(b, -t))};
}
__device__ DD dv_add(DD a, DD b) {
  const DD s = dv_sum(a.h, b.h);
  return dv_sum(s.h, __dadd_rn(s.l, __dadd_rn(a.l, b.l)));
}
__device__ DD dv_mul(DD a, DD b) {
  const double p = __dmul_rn(a.h, b.h);
  return dv_sum(p, __fma_rn(a.h, b.l, __fma_rn(a.l, b.h, __fma_rn(a.h, b.h, -p))));
}
__device__ DD dv_div(double a, double b) {
  const double q = __ddiv_rn(a, b);
  return dv_sum(q, __ddiv_rn(__fma_rn(-q, b, a), b));
}
// ln f = 2 (z + z^3 / 3 + ...), z = (f - 1) / (f + 1), for f in [1/2, 1] of few bits: z^2 <= 1/9, 32 terms to
// 2^-100
__device__ DD dv_log(double f) {
  const DD z = dv_div(f - 1.0, f + 1.0), z2 = dv_mul(z, z);
  DD s = {0.0, 0.0};
  for (int n = 63; n >= 1; n -= 2) s = dv_add(dv_mul(s, z2), dv_div(2.0, n));
  return dv_mul(s, z);
}
__global__ void k_log_tables(LogTables* t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const auto lead = [](DD v) { return rint(v.h * 0x1p42) * 0x1p-42; };
  if (i < LOG_M) {
    // (the first and the last interval have f = 1 and 1/2, where the sums for x around 1 vanish)
    const int hi = __double2hiint(i == 0 ? 1.0 : (i == LOG_M - 1 ? 0.5 : 1.0 / (1.0 + (i + 0.5) / LOG_M)));
    const DD v = dv_log(__hiloint2double(hi, 0));
    const double a = lead(v);
    t->f[i] = hi;
    t->y[i] = 1.0 - a;
    t->yt[i] = -(float)((v.h - a) + v.l);
  }
  if (i < LOG_K) {
    const DD v = dv_mul(dv_log(0.5), {1023.0 - i, 0.0});
    const double a = lead(v);
    t->k[i] = a;
    t->kt[i] = (float)((v.h - a) + v.l);
  }
}
// FP64 <-> FP32 by integer operations (the conversion instructions run at the FP64 pipe's rate): to the
// nearest, for values in FP32's normal range or zero; exact (zero becomes 2^-127)
__device__ __forceinline__ float to_f32(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) + 0x10000000ull;
  const int hi = (int)(b >> 32);
  const unsigned e = (unsigned)max((hi & 0x7fffffff) - 0x38000000, 0);
  return __int_as_float((int)__funnelshift_l((unsigned)b, e, 3) | (hi & 0x80000000));
}
__device__ __forceinline__ double to_f64(float v) {
  const int b = __float_as_int(v);
  return __hiloint2double((int)(((unsigned)(b & 0x7fffffff) >> 3) + 0x38000000u) | (b & 0x80000000), b << 29);
}
// 1 + ln max(x, delta), delta > 0; a NaN stays a NaN.  Positive doubles compare like their bits (an FP64
// comparison would take the pipe).
__device__ __forceinline__ double guarded_log1(double x, double delta, const LogTables* tab) {
  constexpr unsigned LO = 0x00100000u, SPAN = ((unsigned)LOG_K << 20) - LO;  // upper words within the tables
  long long bits = __double_as_longlong(x);
  const long long lo = __double_as_longlong(delta);
  if ((unsigned)(bits >> 32) - LO >= SPAN) {
    x = x < delta ? delta : x;
    bits = __double_as_longlong(x);
    if ((unsigned)(bits >> 32) - LO >= SPAN) return log(x) + 1.0;
  }
  bits = bits < lo ? lo : bits;
  const unsigned hi = (unsigned)(bits >> 32);
  if (hi - LO >= SPAN) return log(__longlong_as_double(bits)) + 1.0;  // a denormal or enormous delta
  const double m = __longlong_as_double((bits & 0x000fffffffffffffLL) | 0x3ff0000000000000LL);
  const int j = (hi >> 9) & (LOG_M - 1);
  const double r = fma(m, __hiloint2double(tab->f[j], 0), -1.0);
  const int rh = __double2hiint(r);
  const double half = __hiloint2double(rh == 0 ? 0 : (rh - 0x00100000) ^ 0x80000000, __double2loint(r));  // -r / 2
  const float s = to_f32(r);
  const float t = fmaf(s * s * s, fmaf(s, fmaf(s, 0.2f, -0.25f), 1.f / 3.f), tab->kt[hi >> 20] + tab->yt[j]);
  return (tab->k[hi >> 20] + tab->y[j]) + (fma(half, r, r) + to_f64(t));
}

// A line of the product rule: the weights of the simplex's vertices in its points -- u and vv of vertices 1 and 2,
// end[k] of vertex 0 and end[2 - k] of vertex D in point k -- and those of its sums A and B (see k_cell_loads_fh)
// against lambda_1, lambda_2 and lambda_0 or lambda_D.
struct FhLine {
  double u, vv, end[3], cu, cv, ca, cb;
};
template <int D>
constexpr FhLine fh_line(int ij) {
  const int i = D == 2 ? ij : ij / 3, j = ij % 3;
  const double root = 3.8729833462074168852;  // sqrt(15), then its rest
  const DD sq = dd_prod(root, root), h = dd_div({root, ((15.0 - sq.h) - sq.l) / (2.0 * root)}, {10.0, 0.0});
  const DD one = {1.0, 0.0}, x[3] = {DD{0.5, 0.0} + DD{-h.h, -h.l}, {0.5, 0.0}, DD{0.5, 0.0} + h};
  const DD u = x[i], w1 = one + DD{-u.h, -u.l}, v = D == 2 ? DD{0.0, 0.0} : x[j], vv = v * w1;
  const DD w2 = w1 + DD{-vv.h, -vv.l};
  DD c = DD{D == 2 ? 2.0 : 6.0, 0.0} * gl_w(i) * w1 * gl_w(0);
  if (D == 3) c = c * gl_w(j) * w2;
  const double gu = gl_grid(u.h), gv = gl_grid(vv.h), gw = (1.0 - gu) - gv, far = gl_grid((w2 * x[0]).h);
  return {gu, gv, {gw - far, 0.5 * gw, far}, (c * u).h, (c * vv).h, 0.5 * (c * w2).h, (c * w2 * h).h};
}
struct FhLines {
  FhLine line[9];
};
template <int D>
constexpr FhLines fh_lines() {
  FhLines t{};
  for (int q = 0; q < (D == 2 ? 3 : 9); ++q) t.line[q] = fh_line<D>(q);
  return t;
}
__constant__ FhLines c_fh_lines[2] = {fh_lines<2>(), fh_lines<3>()};

// eload as k_cell_loads, f' of the Flory-Huggins energy by the product rule: along the innermost direction the
// hat functions are linear.  With f' at a line's points f_0, f_1, f_2, E = f_0 + f_2, A = E + 8/5 f_1 (5/18 A is
// the line's integral) and B = f_2 - f_0 (its moment is 5/18 (A / 2 + h B), h = sqrt(15) / 10).  109 FP64
// instructions for a line's nine logarithms and six values of f' (144 a point with the hat functions tabulated and
// CUDA's log).  f' is summed up at each point, where its large terms cancel: the three logarithms' integrals, summed
// apart and combined at the end, saved nine instructions a line and left three to six times the error.  128 x 128 x
// 32 cells: 19.5 ms at first, 6.1 ms now.  A thread takes a simplex; the simplices' corner values are added in
// shared memory in simplex order, where the tables are as well.
// CB cells per block.  Three blocks of 192 threads per SM: 32 cells of six tetrahedra, 96 of two triangles
// (512 x 512 369 us, a fifth more with 32 cells); 2D meshes of at most two blocks of 32 cells per SM take those
// (64 x 64 29 us, a tenth more with 96 cells).
template <int D, int CB>
constexpr int fh_smem() {
  return (int)(sizeof(LogTables) + sizeof(double2) * CellSimplices<D>::NT * (D + 1) * CB);
}
template <int D, int CB>
__global__ void __launch_bounds__(CB* CellSimplices<D>::NT, 3) k_cell_loads_fh(const MeshPod m, const FhCoef F,
                                                                             const LogTables* __restrict__ tables,
                                                                             const double* pp, const double* pn,
                                                                             int ld, double2* __restrict__ eload) {
  using S = CellSimplices<D>;
  extern __shared__ __align__(16) unsigned char fh_raw[];
  LogTables* tab = reinterpret_cast<LogTables*>(fh_raw);
  double2(*part)[D + 1][CB] = reinterpret_cast<double2(*)[D + 1][CB]>(fh_raw + sizeof(LogTables));
  for (int e = threadIdx.x; e < (int)(sizeof(LogTables) / 16); e += blockDim.x)
    reinterpret_cast<uint4*>(tab)[e] = reinterpret_cast<const uint4*>(tables)[e];
  __syncthreads();
  // one simplex per warp: uniform corners
  const int t = (threadIdx.x >> 5) % S::NT, in = (threadIdx.x >> 5) / S::NT * 32 + (threadIdx.x & 31);
  for (int c0 = blockIdx.x * CB; c0 < m.C; c0 += gridDim.x * CB) {
    const int cell = c0 + in;
    if (cell < m.C) {
      const int* ev = m.elems + ((size_t)cell * S::NT + t) * (D + 1);
      double P[D + 1], Q[D + 1];
#pragma unroll
      for (int a = 0; a <= D; ++a) {
        P[a] = pp[(size_t)ld * ev[a]];
        Q[a] = pn[(size_t)ld * ev[a]];
      }
      double Gp[D + 1], Gn[D + 1];
#pragma unroll
      for (int a = 0; a <= D; ++a) Gp[a] = Gn[a] = 0.0;
#pragma unroll 1
      for (int ij = 0; ij < (D == 2 ? 3 : 9); ++ij) {
        const FhLine& q = c_fh_lines[D - 2].line[ij];
        // positive weights only, so that small concentrations beside large ones keep their relative precision,
        // which their logarithms need
        double pc = q.u * P[1], nc = q.u * Q[1];
        if (D == 3) {
          pc = fma(q.vv, P[2], pc);
          nc = fma(q.vv, Q[2], nc);
        }
        double fp[3], fn[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double p = fma(q.end[k], P[0], fma(q.end[2 - k], P[D], pc));
          const double n = fma(q.end[k], Q[0], fma(q.end[2 - k], Q[D], nc));
          const double ls = guarded_log1(1.0 - p - n, F.delta, tab);
          fp[k] = fma(F.inv_np, guarded_log1(p, F.delta, tab),
                      fma(-F.inv_ns, ls, fma(-2.0 * F.chi_ps, p, fma(F.mix, n, F.chi_ps))));
          fn[k] = fma(F.inv_nn, guarded_log1(n, F.delta, tab),
                      fma(-F.inv_ns, ls, fma(-2.0 * F.chi_ns, n, fma(F.mix, p, F.chi_ns))));
        }
        const auto sums = [&](const double (&f)[3], double (&G)[D + 1]) {
          const double A = fma(1.6, f[1], f[0] + f[2]), B = f[2] - f[0];
          G[0] = fma(q.ca, A, fma(-q.cb, B, G[0]));
          G[1] = fma(q.cu, A, G[1]);
          if (D == 3) G[2] = fma(q.cv, A, G[2]);
          G[D] = fma(q.ca, A, fma(q.cb, B, G[D]));
        };
        sums(fp, Gp);
        sums(fn, Gn);
      }
      // mix_lo int phi lambda_i = mix_lo (<phi> + phi_i) / ((d+1)(d+2)), in units of |T|
      constexpr double q2 = 1.0 / ((D + 1) * (D + 2));
      double Sp = 0.0, Sq = 0.0;
#pragma unroll
      for (int a = 0; a <= D; ++a) {
        Sp += P[a];
        Sq += Q[a];
      }
      const double vol = m.vol[(size_t)cell * S::NT + t], lo = F.mix_lo * q2;
#pragma unroll
      for (int a = 0; a <= D; ++a)
        part[t][a][in] = make_double2(vol * fma(lo, Sq + Q[a], Gp[a]), vol * fma(lo, Sp + P[a], Gn[a]));
    }
    __syncthreads();
    cell_sums<D, CB>(part, c0, m.C, eload);
    __syncthreads();  // before the next cells' values
  }
}

// the Flory-Huggins load's logarithm tables, once per system, and its shared-memory limits
static ch_status log_tables(ch_system_s* s, cudaStream_t st) {
  LogTables* t = nullptr;
  CH_TRY(s->mem.get(&t, 1));
  s->log_tables = t;
  k_log_tables<<<blocks_for(std::max(LOG_M, LOG_K)), TPB, 0, st>>>(t);
  CH_LAUNCHED();
  const auto limit = [](auto kern, int bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  CH_CUDA(limit(k_cell_loads_fh<2, 32>, fh_smem<2, 32>()));
  CH_CUDA(limit(k_cell_loads_fh<2, 96>, fh_smem<2, 96>()));
  CH_CUDA(limit(k_cell_loads_fh<3, 32>, fh_smem<3, 32>()));
  return CH_OK;
}

template <int D>
__device__ void node_loads(const MeshPod& m, const LoadCoef& L, const double2* __restrict__ eload,
                           const double* pp, const double* pn, int ld, int v, double* Fp, double* Fn,
                           double* Gp, double* Gn) {
  double fp = 0.0, fn = 0.0;
  const CellGrid G = m.grid[m.node_run[v]];
  const int l = v - G.node0, x = l % (G.nx + 1), yz = l / (G.nx + 1), y = yz % (G.ny + 1), z = yz / (G.ny + 1);
  constexpr int NC = CellSimplices<D>::NC;
#pragma unroll
  for (int c = NC - 1; c >= 0; --c) {  // cells in increasing order: the node is their corner c
    const int cx = x - (c & 1), cy = y - ((c >> 1) & 1), cz = z - (c >> 2);
    if (cx < 0 || cx >= G.nx || cy < 0 || cy >= G.ny || (D == 3 && (cz < 0 || cz >= G.nz))) continue;
    const double2 e = eload[((size_t)G.cell0 + cx + (size_t)G.nx * (cy + (size_t)G.ny * (D == 3 ? cz : 0))) * NC + c];
    fp += e.x;
    fn += e.y;
  }
  *Fp = fp;
  *Fn = fn;
  double gp = 0.0, gn = 0.0;
  if (L.bc) {
    constexpr int DF = D - 1;
    constexpr double f1 = 1.0 / (DF + 1);                 // int lambda_i / |F|
    constexpr double f2 = 1.0 / ((DF + 1) * (DF + 2));    // int lambda_a lambda_i / |F|, a != i
    constexpr double f3 = (D == 2) ? 1.0 / 24.0 : 1.0 / 60.0;  // (d-1)!/(d+2)!
    if (L.bw) {
      // Gamma_b, patterned: int p_s (g + 2 h phi) lambda_i = g W1_i + 2 h sum_a phi_a W2_ai
      for (int q = m.n2b_ptr[v]; q < m.n2b_ptr[v + 1]; ++q) {
        const int f = m.n2b[q];
        const int* fv = m.bot + D * f;
        const double* Wp = L.bw + (size_t)f * 2 * (D + D * D);
        const double* Wn = Wp + D + D * D;
        int li = 0;
        for (int a = 0; a < D; ++a)
          if (fv[a] == v) li = a;
        double sp = 0.0, sn = 0.0;
        for (int a = 0; a < D; ++a) {
          sp += pp[(size_t)ld * fv[a]] * Wp[D + a * D + li];
          sn += pn[(size_t)ld * fv[a]] * Wn[D + a * D + li];
        }
        gp += L.gp * Wp[li] + 2.0 * L.hp * sp;
        gn += L.gn * Wn[li] + 2.0 * L.hn * sn;
      }
    } else {
      for (int q = m.n2b_ptr[v]; q < m.n2b_ptr[v + 1]; ++q) {  // Gamma_b: int (g + 2 h phi) lambda_i
        const int f = m.n2b[q];
        const int* fv = m.bot + D * f;
        double Sp = 0, Sq = 0, pi = 0, qi = 0;
        for (int a = 0; a < D; ++a) {
          Sp += pp[(size_t)ld * fv[a]];
          Sq += pn[(size_t)ld * fv[a]];
          if (fv[a] == v) {
            pi = pp[(size_t)ld * fv[a]];
            qi = pn[(size_t)ld * fv[a]];
          }
        }
        const double ar = m.bvol[f];
        gp += ar * (L.gp * f1 + 2.0 * L.hp * f2 * (Sp + pi));
        gn += ar * (L.gn * f1 + 2.0 * L.hn * f2 * (Sq + qi));
      }
    }
    for (int q = m.n2t_ptr[v]; q < m.n2t_ptr[v + 1]; ++q) {  // Gamma_t: k int phi phi_s lambda_i
      const int f = m.n2t[q];
      const int* fv = m.top + D * f;
      double Sp = 0, Sq = 0, Ss = 0, Sps = 0, Sqs = 0, pi = 0, qi = 0, si = 0;
      for (int a = 0; a < D; ++a) {
        const double x = pp[(size_t)ld * fv[a]], y = pn[(size_t)ld * fv[a]], s = 1.0 - x - y;
        Sp += x;
        Sq += y;
        Ss += s;
        Sps += x * s;
        Sqs += y * s;
        if (fv[a] == v) {
          pi = x;
          qi = y;
          si = s;
        }
      }
      const double ar = m.tvol[f] * L.kev * f3;
      gp += ar * (Sp * Ss + Sps + pi * Ss + si * Sp + 2.0 * pi * si);
      gn += ar * (Sq * Ss + Sqs + qi * Ss + si * Sq + 2.0 * qi * si);
    }
  }
  *Gp = gp;
  *Gn = gn;
}

static LoadCoef load_coef(const ch_params& p, int dim) {
  LoadCoef L;
  L.cubic = p.potential == 2 ? 0.0 : 7.0 / (dim == 2 ? 360.0 : 840.0);
  L.cs = p.potential == 0 ? 0.2 / (dim == 2 ? 12.0 : 20.0) : 0.0;
  L.bc = p.bc_mode;
  L.gp = p.g_p;
  L.gn = p.g_nfa;
  L.hp = p.h_p;
  L.hn = p.h_nfa;
  L.kev = p.evap_sign * p.k_evap;
  L.bw = nullptr;
  return L;
}

template <int D>
__global__ void k_loads(const MeshPod m, LoadCoef L, const double2* eload, const double* pp,
                        const double* pn, int ld, double* Fp, double* Fn, double* Gp, double* Gn) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= m.N) return;
  double a, b, c, d;
  node_loads<D>(m, L, eload, pp, pn, ld, v, &a, &b, &c, &d);
  if (Fp) Fp[v] = a;
  if (Fn) Fn[v] = b;
  if (Gp) Gp[v] = c;
  if (Gn) Gn[v] = d;
}

// b (N x 4) = (M phi_p + tau g_p, M phi_n + tau g_n, -c F_p, -c F_n)   (Eq. (13) -> Eq. (14))
template <int D>
__global__ void k_rhs(const MeshPod m, LoadCoef L, const double2* eload, const LatOperator A, const int* rowptr,
                      const int* col, const double* valM, const double* pp, const double* pn, int ld,
                      double tau, double c, double* b) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= m.N) return;
  double Fp, Fn, Gp, Gn;
  node_loads<D>(m, L, eload, pp, pn, ld, v, &Fp, &Fn, &Gp, &Gn);
  double mp = 0.0, mn = 0.0;
  if (A.tab) {
    constexpr int ND = D == 2 ? 7 : 15;
    const int id = lat_id(A.L, v);
    const int2 w = A.L.wh[id];
    const double* t = A.tab + (size_t)id * LatAxes<ND>::TS;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      if (__double2hiint(t[d]) == 0) continue;  // (as lat_apply_A)
      const int j = v + lat_off(ND, d, w.x, w.y);
      mp = fma(t[d], pp[(size_t)ld * j], mp);
      mn = fma(t[d], pn[(size_t)ld * j], mn);
    }
  } else {
    for (int q = rowptr[v]; q < rowptr[v + 1]; ++q) {
      const int j = col[q];
      mp = fma(valM[q], pp[(size_t)ld * j], mp);
      mn = fma(valM[q], pn[(size_t)ld * j], mn);
    }
  }
  double4_32a out;
  out.x = mp + tau * Gp;
  out.y = mn + tau * Gn;
  out.z = -c * Fp;
  out.w = -c * Fn;
  reinterpret_cast<double4_32a*>(b)[v] = out;
}

// Per-cell load contributions into s->eload (the system's scratch: calls on one system must not overlap
// on the GPU).  Algorithmic bytes: the vertex values gathered, element indices and measures, the
// contributions written.
static void cell_loads(const ch_system_s* s, const MeshPod& m, const LoadCoef& L, const double* pp,
                       const double* pn, int ld, cudaStream_t st) {
  const double C = m.C, nc = m.dim == 2 ? 4 : 8, nt = m.dim == 2 ? 2 : 6, d1 = m.dim + 1;
  const double bytes = C * (nc * (4.0 + 16.0 + 16.0) + 8.0);
  if (s->p.potential == 3) {
    const ch_params& p = s->p;
    const FhCoef F = fh_coef(p);
    ProfScope ps(st, K_ELEM_LOADS, 0, bytes, C * nt * (m.dim == 2 ? 9 : 27) * 38.0);
    const LogTables* tab = static_cast<const LogTables*>(s->log_tables);
    if (m.dim == 3)
      k_cell_loads_fh<3, 32><<<std::min(blocks_for(m.C, 32), 3 * 152), 192, fh_smem<3, 32>(), st>>>(m, F, tab, pp, pn,
                                                                                                  ld, s->eload);
    else if (m.C > 2 * 152 * 32)
      k_cell_loads_fh<2, 96><<<std::min(blocks_for(m.C, 96), 3 * 152), 192, fh_smem<2, 96>(), st>>>(m, F, tab, pp, pn,
                                                                                                  ld, s->eload);
    else
      k_cell_loads_fh<2, 32><<<blocks_for(m.C, 32), 64, fh_smem<2, 32>(), st>>>(m, F, tab, pp, pn, ld, s->eload);
    return;
  }
  ProfScope ps(st, K_ELEM_LOADS, 0, bytes, C * nt * (40.0 + 10.0 * d1));
  if (m.dim == 2)
    k_cell_loads<2><<<blocks_for(m.C, 128), 128, 0, st>>>(m, L, pp, pn, ld, s->eload);
  else if (m.C <= 152 * 64)  // two warps of cells per SM, twelve of simplices
    k_cell_loads_split<3><<<blocks_for(m.C, 32), 192, 0, st>>>(m, L, pp, pn, ld, s->eload);
  else
    k_cell_loads<3><<<blocks_for(m.C, 128), 128, 0, st>>>(m, L, pp, pn, ld, s->eload);
}

ch_status loads(const ch_system_s* s, const double* pp, const double* pn, double* Fp, double* Fn,
                double* gp, double* gn, cudaStream_t st) {
  const MeshPod m = mesh_pod(s->mesh);
  LoadCoef L = load_coef(s->p, s->mesh->dim);
  L.bw = s->bw;
  cell_loads(s, m, L, pp, pn, 1, st);
  ProfScope ps(st, K_LOADS, 0, 16.0 * m.N + 32.0 * m.N, 0.0);
  if (m.dim == 2)
    k_loads<2><<<blocks_for(m.N), TPB, 0, st>>>(m, L, s->eload, pp, pn, 1, Fp, Fn, gp, gn);
  else
    k_loads<3><<<blocks_for(m.N), TPB, 0, st>>>(m, L, s->eload, pp, pn, 1, Fp, Fn, gp, gn);
  CH_LAUNCHED();
  return CH_OK;
}

ch_status rhs_strided(const ch_system_s* s, const double* pp, const double* pn, int ld, double* b,
                      cudaStream_t st) {
  const MeshPod m = mesh_pod(s->mesh);
  LoadCoef L = load_coef(s->p, s->mesh->dim);
  L.bw = s->bw;
  cell_loads(s, m, L, pp, pn, ld, st);
  // phi read + b written + M (values, columns, row pointers) + the cells' contributions gathered
  ProfScope ps(st, K_RHS, 0, 48.0 * m.N + 12.0 * s->nnz + 4.0 * m.N + m.C * (m.dim == 2 ? 64.0 : 128.0),
               2.0 * s->nnz);
  if (m.dim == 2)
    k_rhs<2><<<blocks_for(m.N), TPB, 0, st>>>(m, L, s->eload, s->lat, s->rowptr, s->col, s->valM, pp, pn, ld,
                                               s->p.tau, s->c, b);
  else
    k_rhs<3><<<blocks_for(m.N), TPB, 0, st>>>(m, L, s->eload, s->lat, s->rowptr, s->col, s->valM, pp, pn, ld,
                                               s->p.tau, s->c, b);
  CH_LAUNCHED();
  return CH_OK;
}

// ---------------------------------------------------------------- block operator of Eq. (14)
// y = A x for both species: per node x = (x1_p, x1_n, x2_p, x2_n),
//   y1 = M x1 + a K x2,  y2 = a K x1 - c M x2.
// One pass over the shared pattern: 8 FMAs per stored entry.
__global__ void k_apply_A(int N, const int* rowptr, const int* col, const double* valM,
                          const double* valK, double a, double c, const double4_32a* x, double4_32a* y) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= N) return;
  double m1p = 0, m1n = 0, m2p = 0, m2n = 0, k1p = 0, k1n = 0, k2p = 0, k2n = 0;
  for (int q = rowptr[v]; q < rowptr[v + 1]; ++q) {
    const int j = col[q];
    const double m = valM[q], k = valK[q];
    const double4_32a z = x[j];
    m1p = fma(m, z.x, m1p);
    m1n = fma(m, z.y, m1n);
    m2p = fma(m, z.z, m2p);
    m2n = fma(m, z.w, m2n);
    k1p = fma(k, z.x, k1p);
    k1n = fma(k, z.y, k1n);
    k2p = fma(k, z.z, k2p);
    k2n = fma(k, z.w, k2n);
  }
  double4_32a out;
  out.x = fma(a, k2p, m1p);
  out.y = fma(a, k2n, m1n);
  out.z = fma(a, k1p, -c * m2p);
  out.w = fma(a, k1n, -c * m2n);
  y[v] = out;
}

// The lattice form: no indices or values but the class id, so the FP64 pipe alone bounds it (54 or 94
// instructions per node).  512 x 512: 27.3 us, 33.6 in CSR form; 3D 128 x 128 x 32: 91, 127 in
// CSR form.  Several classes along an axis cost little (in a run of launches: 512 x 512 and 511 x 509 29.3 us, 128 x
// 128 x 32 93 and 127 x 129 x 33 95).
template <int ND>
__global__ void __launch_bounds__(128) k_apply_A_lat(LatOperator A, int N, const double4_32a* __restrict__ x,
                                                     double4_32a* __restrict__ y) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < N) y[v] = lat_apply_A<ND>(A, v, x);
}

ch_status apply_A(const ch_system_s* s, const double* x, double* y, cudaStream_t st) {
  const double4_32a* x4 = reinterpret_cast<const double4_32a*>(x);
  double4_32a* y4 = reinterpret_cast<double4_32a*>(y);
  if (s->lat.tab) {
    const double f = s->mesh->dim == 2 ? 54.0 : 94.0;
    ProfScope ps(st, K_APPLY_A, 0, 66.0 * s->N, f * s->N);
    if (s->mesh->dim == 2) k_apply_A_lat<7><<<blocks_for(s->N, 128), 128, 0, st>>>(s->lat, s->N, x4, y4);
    else k_apply_A_lat<15><<<blocks_for(s->N, 128), 128, 0, st>>>(s->lat, s->N, x4, y4);
  } else {
    ProfScope ps(st, K_APPLY_A, 0, 20.0 * s->nnz + 4.0 * (s->N + 1) + 64.0 * s->N, 8.0 * s->nnz + 4.0 * s->N);
    k_apply_A<<<blocks_for(s->N), TPB, 0, st>>>(s->N, s->rowptr, s->col, s->valM, s->valK, s->a, s->c, x4, y4);
  }
  CH_LAUNCHED();
  return CH_OK;
}

}  // namespace ch
