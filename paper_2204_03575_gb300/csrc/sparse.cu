// Sparse-structure primitives used at set-up: scans, incidence lists, transpose and a
// deterministic sparse matrix product (Galerkin products of the AMG set-up).
#include <cstdarg>

#include "ch_internal.cuh"

namespace ch {

static thread_local std::string g_err;

void set_error(const char* fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
}

const char* last_error() { return g_err.c_str(); }

// ---------------------------------------------------------------- exclusive scan
// Row pointers from counts: tile sums, their scan (int64, one block, tile after tile), then the tiles' own
// scans on top.
constexpr int SCAN_IT = 4;
constexpr int SCAN_TILE = TPB * SCAN_IT;

// exclusive scan of one tile of values v (thread-contiguous) within the block; returns the tile's sum
__device__ __forceinline__ int64_t scan_tile(int64_t (&v)[SCAN_IT]) {
  __shared__ int64_t warp_tot[TPB / 32 + 1];
  int64_t tsum = 0;
#pragma unroll
  for (int k = 0; k < SCAN_IT; ++k) tsum += v[k];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t x = tsum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  int64_t excl = x - tsum, total = 0;
#pragma unroll
  for (int q = 0; q < TPB / 32; ++q) {
    if (q < w) excl += warp_tot[q];
    total += warp_tot[q];
  }
#pragma unroll
  for (int k = 0; k < SCAN_IT; ++k) {
    const int64_t t = v[k];
    v[k] = excl;
    excl += t;
  }
  return total;
}

__global__ void k_scan_sums(const int* counts, int n, int64_t* sums) {
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_IT;
  int64_t v[SCAN_IT];
#pragma unroll
  for (int k = 0; k < SCAN_IT; ++k) v[k] = base + k < n ? counts[base + k] : 0;
  const int64_t t = scan_tile(v);
  if (threadIdx.x == 0) sums[blockIdx.x] = t;
}

// in place; one block: the tiles one after another (n tile sums; n <= 2^31 / 1024), total at d[n]
__global__ void k_scan_totals(int64_t* d, int n) {
  __shared__ int64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t b = 0; b < n; b += SCAN_TILE) {
    const int64_t base = b + (int64_t)threadIdx.x * SCAN_IT;
    int64_t v[SCAN_IT];
#pragma unroll
    for (int k = 0; k < SCAN_IT; ++k) v[k] = base + k < n ? d[base + k] : 0;
    const int64_t t = scan_tile(v), c = carry;
#pragma unroll
    for (int k = 0; k < SCAN_IT; ++k)
      if (base + k < n) d[base + k] = c + v[k];
    __syncthreads();
    if (threadIdx.x == 0) carry = c + t;
    __syncthreads();
  }
  if (threadIdx.x == 0) d[n] = carry;
}

__global__ void k_scan_rows(const int* counts, int n, const int64_t* offs, int* rowptr) {
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_IT;
  int64_t v[SCAN_IT];
#pragma unroll
  for (int k = 0; k < SCAN_IT; ++k) v[k] = base + k < n ? counts[base + k] : 0;
  scan_tile(v);
  const int64_t o = offs[blockIdx.x];
#pragma unroll
  for (int k = 0; k < SCAN_IT; ++k)
    if (base + k < n) rowptr[base + k] = (int)(o + v[k]);
  if (blockIdx.x == 0 && threadIdx.x == 0) rowptr[n] = (int)offs[gridDim.x];
}

ch_status scan_i32_to_rowptr(const int* counts, int* rowptr, int n, int64_t* total, cudaStream_t st,
                             Alloc& tmp) {
  int64_t* t = nullptr;
  const int nt = n > 0 ? (int)(((int64_t)n + SCAN_TILE - 1) / SCAN_TILE) : 1;
  CH_TRY(tmp.get(&t, (size_t)nt + 1));
  k_scan_sums<<<nt, TPB, 0, st>>>(counts, n, t);
  k_scan_totals<<<1, TPB, 0, st>>>(t, nt);
  k_scan_rows<<<nt, TPB, 0, st>>>(counts, n, t, rowptr);
  CH_LAUNCHED();
  int64_t tot = 0;
  CH_CUDA(cudaMemcpyAsync(&tot, t + nt, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  CH_CUDA(cudaStreamSynchronize(st));
  if (tot > 2147483647LL) {
    set_error("sparse structure with %lld entries exceeds int32 indexing", (long long)tot);
    return CH_ERR_INTERNAL;
  }
  if (total) *total = tot;
  return CH_OK;
}

// ---------------------------------------------------------------- incidence lists
__global__ void k_count_keys(const int* items, int64_t nent, int* cnt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nent) atomicAdd(&cnt[items[i]], 1);
}
__global__ void k_fill_keys(const int* items, int64_t nent, int k, const int* ptr, int* cur,
                            int* list) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nent) {
    const int key = items[i];
    const int slot = atomicAdd(&cur[key], 1);
    list[ptr[key] + slot] = (int)(i / k);
  }
}
// insertion sort of each list (lists are short: node -> incident simplices)
__global__ void k_sort_lists(const int* ptr, int* list, int nkeys) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nkeys) return;
  const int b = ptr[r], e = ptr[r + 1];
  for (int i = b + 1; i < e; ++i) {
    const int v = list[i];
    int j = i - 1;
    while (j >= b && list[j] > v) {
      list[j + 1] = list[j];
      --j;
    }
    list[j + 1] = v;
  }
}

ch_status build_incidence(const int* items, int nitems, int k, int nkeys, int** ptr, int** list,
                          cudaStream_t st, Alloc& mem) {
  const int64_t nent = (int64_t)nitems * k;
  Alloc tmp;
  int* cnt = nullptr;
  CH_TRY(tmp.get(&cnt, (size_t)nkeys));
  CH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * nkeys, st));
  if (nent > 0) {
    k_count_keys<<<blocks_for(nent), TPB, 0, st>>>(items, nent, cnt);
    CH_LAUNCHED();
  }
  CH_TRY(mem.get(ptr, (size_t)nkeys + 1));
  int64_t tot = 0;
  CH_TRY(scan_i32_to_rowptr(cnt, *ptr, nkeys, &tot, st, tmp));
  CH_TRY(mem.get(list, (size_t)tot));
  CH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * nkeys, st));
  if (nent > 0) {
    k_fill_keys<<<blocks_for(nent), TPB, 0, st>>>(items, nent, k, *ptr, cnt, *list);
    CH_LAUNCHED();
  }
  k_sort_lists<<<blocks_for(nkeys), TPB, 0, st>>>(*ptr, *list, nkeys);
  CH_LAUNCHED();
  CH_CUDA(cudaStreamSynchronize(st));  // tmp is released on return
  return CH_OK;
}

// ---------------------------------------------------------------- transpose
__global__ void k_col_count(const int* col, int64_t nnz, int* cnt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nnz) atomicAdd(&cnt[col[i]], 1);
}
__global__ void k_transpose_fill(Csr<double> A, const int* bptr, int* cur, int* bcol, double* bval) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= A.nrows) return;
  for (int p = A.rowptr[r]; p < A.rowptr[r + 1]; ++p) {
    const int c = A.col[p];
    const int q = bptr[c] + atomicAdd(&cur[c], 1);
    bcol[q] = r;
    bval[q] = A.val[p];
  }
}
// Sorts each row's (distinct) columns, one warp per row: rows of at most SORT_MAX entries are ranked
// in shared memory (each lane counts the columns below its own), longer ones by insertion.
constexpr int SORT_MAX = 256, SORT_WARPS = 8;
__global__ void __launch_bounds__(32 * SORT_WARPS) k_sort_rows(const int* ptr, int* col, double* val, int n) {
  __shared__ int sc[SORT_WARPS][SORT_MAX];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * SORT_WARPS + w;
  if (r >= n) return;
  const int b = ptr[r], len = ptr[r + 1] - b;
  if (len <= SORT_MAX) {
    constexpr int PER = SORT_MAX / 32;
    int c[PER], rank[PER];
    double v[PER];
#pragma unroll
    for (int t = 0; t < PER; ++t) {
      const int e = 32 * t + lane;
      rank[t] = 0;
      if (e < len) {
        c[t] = col[b + e];
        v[t] = val[b + e];
        sc[w][e] = c[t];
      }
    }
    __syncwarp();
    for (int j = 0; j < len; ++j) {
      const int kj = sc[w][j];
#pragma unroll
      for (int t = 0; t < PER; ++t)
        if (32 * t < len) rank[t] += kj < c[t];
    }
#pragma unroll
    for (int t = 0; t < PER; ++t)
      if (32 * t + lane < len) {
        col[b + rank[t]] = c[t];
        val[b + rank[t]] = v[t];
      }
    return;
  }
  if (lane != 0) return;
  for (int i = b + 1; i < b + len; ++i) {
    const int c = col[i];
    const double v = val[i];
    int j = i - 1;
    while (j >= b && col[j] > c) {
      col[j + 1] = col[j];
      val[j + 1] = val[j];
      --j;
    }
    col[j + 1] = c;
    val[j + 1] = v;
  }
}

ch_status transpose(const Csr<double>& A, Csr<double>* B, cudaStream_t st, Alloc& mem) {
  Alloc tmp;
  int* cnt = nullptr;
  CH_TRY(tmp.get(&cnt, (size_t)A.ncols));
  CH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * A.ncols, st));
  if (A.nnz > 0) {
    k_col_count<<<blocks_for(A.nnz), TPB, 0, st>>>(A.col, A.nnz, cnt);
    CH_LAUNCHED();
  }
  B->nrows = A.ncols;
  B->ncols = A.nrows;
  CH_TRY(mem.get(&B->rowptr, (size_t)B->nrows + 1));
  int64_t tot = 0;
  CH_TRY(scan_i32_to_rowptr(cnt, B->rowptr, B->nrows, &tot, st, tmp));
  B->nnz = tot;
  CH_TRY(mem.get(&B->col, (size_t)tot));
  CH_TRY(mem.get(&B->val, (size_t)tot));
  CH_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int) * A.ncols, st));
  k_transpose_fill<<<blocks_for(A.nrows), TPB, 0, st>>>(A, B->rowptr, cnt, B->col, B->val);
  CH_LAUNCHED();
  k_sort_rows<<<blocks_for(B->nrows, SORT_WARPS), 32 * SORT_WARPS, 0, st>>>(B->rowptr, B->col, B->val, B->nrows);
  CH_LAUNCHED();
  CH_CUDA(cudaStreamSynchronize(st));
  return CH_OK;
}

// ---------------------------------------------------------------- C = A * B
// Row i of C is the sum of the rows B_k, k in row i of A, scaled by a_ik.  One warp per row keeps the
// row's columns (and, when filling, its values) in a hash table in shared memory; it takes the entries
// of A's row in order and lets the lanes take the entries of B_k, whose columns are distinct, so every
// column's terms are added in the order of A's row: the product is bitwise reproducible.  The columns
// are then ranked against one another (each lane counts the smaller ones) and written in order.
//
// The table holds CAP columns and is never filled beyond 3/4.  The counting pass takes the smallest CAP
// that the longest row's number of terms (or B's column count) cannot overfill, 4096 at most, and
// stops at a row with more than 3072 columns; the product then takes the heap kernels below.  The
// filling pass knows the counts and takes the smallest CAP that fits them.  Measured on the twelve
// products of a 256 x 256 set-up: both passes 0.65 ms, against 27.1 ms for the one-thread-per-row merge.
__global__ void k_product_counts(Csr<double> A, const int* bptr, int* most) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  int64_t n = 0;
  if (i < A.nrows)
    for (int q = A.rowptr[i]; q < A.rowptr[i + 1]; ++q) n += bptr[A.col[q] + 1] - bptr[A.col[q]];
  int m = n > 0x7fffffff ? 0x7fffffff : (int)n;
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(most, m);
}

template <int CAP>
__device__ __forceinline__ int hash_slot(int* key, int c, int* added) {
  int h = (int)(((uint32_t)c * 2654435761u) >> 7) & (CAP - 1);
  for (;;) {  // ends: a table is never filled beyond 3/4 and one warp's worth
    const int old = atomicCAS(&key[h], -1, c);
    *added = old == -1;
    if (old == -1 || old == c) return h;
    h = (h + 1) & (CAP - 1);
  }
}

template <int CAP>
constexpr int spgemm_warps() { return CAP <= 64 ? 8 : (CAP <= 512 ? 4 : (CAP <= 2048 ? 2 : 1)); }

// counting (FILL = false): cnt[i], and most[0] = the largest count, most[1] = 1 after a row that overfills
template <int CAP, bool FILL>
__global__ void __launch_bounds__(32 * spgemm_warps<CAP>()) k_spgemm_hash(Csr<double> A, Csr<double> B, int* cnt,
                                                                          int* most, const int* cptr, int* ccol,
                                                                          double* cval) {
  constexpr int NW = spgemm_warps<CAP>();
  extern __shared__ __align__(16) unsigned char sp_smem[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double* val = reinterpret_cast<double*>(sp_smem) + (FILL ? w * CAP : 0);
  int* key = reinterpret_cast<int*>(sp_smem + (FILL ? sizeof(double) * NW * CAP : 0)) + w * CAP;
  const int i = blockIdx.x * NW + w;
  if (i >= A.nrows) return;  // whole warp
  for (int h = lane; h < CAP; h += 32) {
    key[h] = -1;
    if (FILL) val[h] = 0.0;
  }
  __syncwarp();
  const int a0 = A.rowptr[i], a1 = A.rowptr[i + 1];
  int held = 0;  // columns in the table (counting)
  for (int base = a0; base < a1; base += 32) {
    // the next 32 entries of A's row and the extents of their rows of B, one per lane
    int p0 = 0, p1 = 0;
    double av = 0.0;
    if (base + lane < a1) {
      const int k = A.col[base + lane];
      if (FILL) av = A.val[base + lane];
      p0 = B.rowptr[k];
      p1 = B.rowptr[k + 1];
    }
    const int m = min(32, a1 - base);
    for (int r = 0; r < m; ++r) {
      const int b0 = __shfl_sync(0xffffffffu, p0, r), b1 = __shfl_sync(0xffffffffu, p1, r);
      const double a = FILL ? __shfl_sync(0xffffffffu, av, r) : 0.0;
      for (int p = b0; p < b1; p += 32) {
        int added = 0;
        if (p + lane < b1) {
          const int h = hash_slot<CAP>(key, B.col[p + lane], &added);
          if (FILL) val[h] = fma(a, B.val[p + lane], val[h]);
        }
        if (!FILL) {
          held += __popc(__ballot_sync(0xffffffffu, added));
          if (held > CAP / 4 * 3) {  // uniform over the warp
            if (lane == 0) most[1] = 1;
            return;
          }
        }
      }
      __syncwarp();
    }
  }
  if (!FILL) {
    if (lane == 0) {
      cnt[i] = held;
      atomicMax(most, held);
    }
    return;
  }
  // compact the occupied slots to the front (slots only move down), then rank
  int n = 0;
  for (int h0 = 0; h0 < CAP; h0 += 32) {
    const int c = key[h0 + lane];
    const double v = val[h0 + lane];
    const unsigned on = __ballot_sync(0xffffffffu, c != -1);
    __syncwarp();
    if (c != -1) {
      const int at = n + __popc(on & ((1u << lane) - 1));
      key[at] = c;
      val[at] = v;
    }
    n += __popc(on);
    __syncwarp();
  }
  const int out = cptr[i];
  for (int e0 = 0; e0 < n; e0 += 128) {  // four columns per lane and sweep over the row
    int c[4], rank[4] = {0, 0, 0, 0};
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int e = e0 + 32 * t + lane;
      c[t] = e < n ? key[e] : -1;
    }
    for (int j = 0; j < n; ++j) {
      const int kj = key[j];
#pragma unroll
      for (int t = 0; t < 4; ++t) rank[t] += kj < c[t];
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int e = e0 + 32 * t + lane;
      if (e < n) {
        ccol[out + rank[t]] = c[t];
        cval[out + rank[t]] = val[e];
      }
    }
  }
}

// The product as a k-way merge, one thread per row with a binary min-heap of (column, run) keys in a
// scratch array laid out like A's entries, so it has no size limit; ties pop in run order, which is
// the order of the sums above.
__device__ __forceinline__ uint64_t mkey(int col, int run) {
  return ((uint64_t)(uint32_t)col << 32) | (uint32_t)run;
}

__device__ void heap_down(uint64_t* h, int n, int i) {
  for (;;) {
    int l = 2 * i + 1, m = i;
    if (l < n && h[l] < h[m]) m = l;
    if (l + 1 < n && h[l + 1] < h[m]) m = l + 1;
    if (m == i) return;
    const uint64_t t = h[i];
    h[i] = h[m];
    h[m] = t;
    i = m;
  }
}

template <bool FILL>
__global__ void k_spgemm_row(Csr<double> A, Csr<double> B, uint64_t* heap, int* cur, int* cnt,
                             const int* cptr, int* ccol, double* cval) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.nrows) return;
  const int a0 = A.rowptr[i], a1 = A.rowptr[i + 1];
  uint64_t* h = heap + a0;
  int* cu = cur + a0;
  int n = 0;
  for (int r = 0; r < a1 - a0; ++r) {
    const int k = A.col[a0 + r];
    const int p = B.rowptr[k];
    cu[r] = p;
    if (p < B.rowptr[k + 1]) h[n++] = mkey(B.col[p], r);
  }
  for (int j = n / 2 - 1; j >= 0; --j) heap_down(h, n, j);
  int out = FILL ? cptr[i] : 0;
  int count = 0, last = -1;
  double acc = 0.0;
  while (n > 0) {
    const uint64_t top = h[0];
    const int c = (int)(top >> 32), r = (int)(top & 0xffffffffu);
    const int p = cu[r];
    if (c != last) {
      if (FILL && last >= 0) {
        ccol[out] = last;
        cval[out] = acc;
        ++out;
      }
      last = c;
      acc = 0.0;
      ++count;
    }
    if (FILL) acc = fma(A.val[a0 + r], B.val[p], acc);
    const int k = A.col[a0 + r];
    const int pn = p + 1;
    cu[r] = pn;
    if (pn < B.rowptr[k + 1]) {
      h[0] = mkey(B.col[pn], r);
    } else {
      h[0] = h[--n];
    }
    heap_down(h, n, 0);
  }
  if (FILL && last >= 0) {
    ccol[out] = last;
    cval[out] = acc;
  }
  if (!FILL) cnt[i] = count;
}

template <int CAP, bool FILL>
static ch_status launch_hash(const Csr<double>& A, const Csr<double>& B, int* cnt, int* most,
                             const Csr<double>* C, cudaStream_t st) {
  constexpr int NW = spgemm_warps<CAP>();
  constexpr int smem = NW * CAP * (int)(sizeof(int) + (FILL ? sizeof(double) : 0));
  if (smem > 48 * 1024)
    CH_CUDA(cudaFuncSetAttribute(k_spgemm_hash<CAP, FILL>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  k_spgemm_hash<CAP, FILL><<<blocks_for(A.nrows, NW), 32 * NW, smem, st>>>(A, B, cnt, most,
                                                                           C ? C->rowptr : nullptr, C ? C->col : nullptr,
                                                                           C ? C->val : nullptr);
  CH_LAUNCHED();
  return CH_OK;
}

template <bool FILL>
static ch_status dispatch_hash(int columns, const Csr<double>& A, const Csr<double>& B, int* cnt, int* most,
                               const Csr<double>* C, cudaStream_t st) {
  if (columns <= 48) return launch_hash<64, FILL>(A, B, cnt, most, C, st);
  if (columns <= 192) return launch_hash<256, FILL>(A, B, cnt, most, C, st);
  if (columns <= 768) return launch_hash<1024, FILL>(A, B, cnt, most, C, st);
  return launch_hash<4096, FILL>(A, B, cnt, most, C, st);
}

ch_status spgemm(const Csr<double>& A, const Csr<double>& B, Csr<double>* C, cudaStream_t st,
                 Alloc& mem) {
  if (A.ncols != B.nrows) {
    set_error("spgemm: inner sizes differ (%d vs %d)", A.ncols, B.nrows);
    return CH_ERR_INTERNAL;
  }
  Alloc tmp;
  int *cnt = nullptr, *most = nullptr;
  CH_TRY(tmp.get(&cnt, (size_t)A.nrows));
  CH_TRY(tmp.get(&most, 2));
  const auto read_most = [&](int (&h)[2]) -> ch_status {
    CH_CUDA(cudaMemcpyAsync(h, most, sizeof(h), cudaMemcpyDeviceToHost, st));
    CH_CUDA(cudaStreamSynchronize(st));
    return CH_OK;
  };
  int h[2] = {0, 0};
  CH_CUDA(cudaMemsetAsync(most, 0, 2 * sizeof(int), st));
  k_product_counts<<<blocks_for(A.nrows), TPB, 0, st>>>(A, B.rowptr, most);
  CH_LAUNCHED();
  CH_TRY(read_most(h));
  const int bound = h[0] < B.ncols ? h[0] : B.ncols;  // no row has more columns
  CH_CUDA(cudaMemsetAsync(most, 0, 2 * sizeof(int), st));
  CH_TRY(dispatch_hash<false>(bound, A, B, cnt, most, nullptr, st));
  CH_TRY(read_most(h));
  const bool hash = h[1] == 0;
  uint64_t* heap = nullptr;
  int* cur = nullptr;
  if (!hash) {
    CH_TRY(tmp.get(&heap, (size_t)A.nnz));
    CH_TRY(tmp.get(&cur, (size_t)A.nnz));
    k_spgemm_row<false><<<blocks_for(A.nrows, 128), 128, 0, st>>>(A, B, heap, cur, cnt, nullptr, nullptr, nullptr);
    CH_LAUNCHED();
  }
  C->nrows = A.nrows;
  C->ncols = B.ncols;
  CH_TRY(mem.get(&C->rowptr, (size_t)C->nrows + 1));
  int64_t tot = 0;
  CH_TRY(scan_i32_to_rowptr(cnt, C->rowptr, C->nrows, &tot, st, tmp));
  C->nnz = tot;
  CH_TRY(mem.get(&C->col, (size_t)tot));
  CH_TRY(mem.get(&C->val, (size_t)tot));
  if (hash) {
    CH_TRY(dispatch_hash<true>(h[0], A, B, nullptr, nullptr, C, st));
  } else {
    k_spgemm_row<true><<<blocks_for(A.nrows, 128), 128, 0, st>>>(A, B, heap, cur, cnt, C->rowptr, C->col, C->val);
    CH_LAUNCHED();
  }
  CH_CUDA(cudaStreamSynchronize(st));
  return CH_OK;
}

}  // namespace ch
