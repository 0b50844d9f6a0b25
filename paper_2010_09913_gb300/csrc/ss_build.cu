// Device-side SlimSell builder (Sections II-D and III-B; SlimChunk split table, Section III-D).
//
//   1. degrees and the sort key (window of sigma vertices, descending degree)
//   2. stable LSD radix sort of (key, vertex) -> perm; ties keep ascending id
//   3. invperm, per-row degree, chunk lengths cl, chunk starts cs (exclusive scan)
//   4. work-item tables: pack items (fixed width) and BFS items (SlimChunk width)
//   5. column-major pack: col[cs_i + j*C + l] = invperm[j-th neighbour of row i*C+l,
//      descending original id], or -1 for padding
#include <cstdarg>
#include <climits>
#include <algorithm>
#include <utility>
#include <vector>

#include "ss_device.cuh"
#include "ss_sort.cuh"

namespace ss {

static thread_local char g_err[512] = "";

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

const char* last_error() { return g_err; }

ss_status cuda_fail(cudaError_t e, const char* what) {
  set_error("CUDA error %s (%s) in %s", cudaGetErrorName(e), cudaGetErrorString(e), what);
  return e == cudaErrorMemoryAllocation ? SS_ERR_OOM : SS_ERR_CUDA;
}

ss_status dmalloc(slimsell_graph* h, void** p, size_t bytes) {
  if (bytes == 0) bytes = 16;
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation && h && drop_planes(h)) {  // what a handle can do without goes first
    cudaGetLastError();
    e = cudaMalloc(p, bytes);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();  // the error is reported here, not by the next launch's check as well
    *p = nullptr;
    return cuda_fail(e, "cudaMalloc");
  }
  if (h) h->device_bytes += (long long)bytes;
  return SS_OK;
}

namespace {
// Several arrays in one device allocation (a handle made 47 cudaMalloc and 47
// cudaFree calls, 3 ms of a 7.5 ms build of Kronecker 22): arrays are announced,
// then placed at 256-byte boundaries of one allocation.
struct Slab {
  std::vector<std::pair<void**, size_t>> want;
  size_t total = 0;
  template <class T>
  void add(T** p, size_t count) {
    want.push_back({(void**)p, total});
    total += (std::max<size_t>(count, 1) * sizeof(T) + 255) / 256 * 256;
  }
  ss_status place(slimsell_graph* h, void** base) {
    ss_status s = dmalloc(h, base, total);
    if (s != SS_OK) return s;
    for (auto& w : want) *w.first = (char*)*base + w.second;
    return SS_OK;
  }
};
}  // namespace

// ---------------------------------------------------------------------------
// Exclusive prefix sum over int64 (three passes: tile sums, scan of sums, tile scans)
// ---------------------------------------------------------------------------

__device__ __forceinline__ long long warp_incl_scan(long long v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    long long t = __shfl_up_sync(SS_FULL_MASK, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// block-wide exclusive scan of one value per thread; returns the block total in *total
__device__ __forceinline__ long long block_excl_scan(long long v, long long* total) {
  __shared__ long long wsum[SCAN_THREADS / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long inc = warp_incl_scan(v);
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    long long s = (lane < SCAN_THREADS / 32) ? wsum[lane] : 0;
    s = warp_incl_scan(s);
    if (lane < SCAN_THREADS / 32) wsum[lane] = s;
  }
  __syncthreads();
  long long before = (w > 0 ? wsum[w - 1] : 0) + inc - v;
  *total = wsum[SCAN_THREADS / 32 - 1];
  __syncthreads();
  return before;
}

__global__ void k_tile_sum(const long long* in, long long n, long long* partial) {
  long long base = (long long)blockIdx.x * SCAN_TILE;
  long long s = 0;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    long long idx = base + (long long)i * SCAN_THREADS + threadIdx.x;
    if (idx < n) s += in[idx];
  }
  long long total;
  block_excl_scan(s, &total);
  if (threadIdx.x == 0) partial[blockIdx.x] = total;
}

__global__ void k_scan_partials(long long* partial, int ntiles) {
  // one block of 1024 threads; each thread owns a contiguous run
  __shared__ long long sums[1024];
  const int t = threadIdx.x;
  const int per = (ntiles + 1023) / 1024;
  const int lo = min(t * per, ntiles), hi = min(lo + per, ntiles);
  long long s = 0;
  for (int i = lo; i < hi; ++i) s += partial[i];
  sums[t] = s;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    long long v = (t >= o) ? sums[t - o] : 0;
    __syncthreads();
    sums[t] += v;
    __syncthreads();
  }
  long long run = sums[t] - s;
  for (int i = lo; i < hi; ++i) {
    long long v = partial[i];
    partial[i] = run;
    run += v;
  }
}

__global__ void k_tile_scan(const long long* in, long long* out, long long n, const long long* partial) {
  __shared__ long long tile[SCAN_TILE];
  long long base = (long long)blockIdx.x * SCAN_TILE;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    long long idx = base + (long long)i * SCAN_THREADS + threadIdx.x;
    tile[i * SCAN_THREADS + threadIdx.x] = (idx < n) ? in[idx] : 0;
  }
  __syncthreads();
  long long s = 0;
  long long* mine = tile + threadIdx.x * SCAN_ITEMS;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) s += mine[i];
  long long total;
  long long run = block_excl_scan(s, &total) + partial[blockIdx.x];
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    long long v = mine[i];
    mine[i] = run;
    run += v;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    long long idx = base + (long long)i * SCAN_THREADS + threadIdx.x;
    if (idx < n) out[idx] = tile[i * SCAN_THREADS + threadIdx.x];
  }
}

// exclusive scan of n int64 values in place; `tmp` must hold ceil(n / SCAN_TILE) entries
ss_status excl_scan(long long* data, long long n, long long* tmp, cudaStream_t st) {
  if (n <= 0) return SS_OK;
  long long ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
  k_tile_sum<<<(unsigned)ntiles, SCAN_THREADS, 0, st>>>(data, n, tmp);
  k_scan_partials<<<1, 1024, 0, st>>>(tmp, (int)ntiles);
  k_tile_scan<<<(unsigned)ntiles, SCAN_THREADS, 0, st>>>(data, data, n, tmp);
  SS_CUDA(cudaGetLastError());
  return SS_OK;
}

// ---------------------------------------------------------------------------
// Stable LSD radix sort of (uint64 key, int32 value), 8-bit digits
// ---------------------------------------------------------------------------

__global__ void k_rs_hist(const unsigned long long* keys, int n, int shift, long long* hist, int nblk) {
  __shared__ unsigned h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  long long base = (long long)blockIdx.x * RS_TILE;
#pragma unroll 4
  for (int i = 0; i < RS_ITEMS; ++i) {
    long long idx = base + (long long)i * RS_THREADS + threadIdx.x;
    if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & 255u], 1u);
  }
  __syncthreads();
  hist[(long long)threadIdx.x * nblk + blockIdx.x] = h[threadIdx.x];
}

__global__ void k_rs_scatter(const unsigned long long* kin, const int* vin, unsigned long long* kout,
                             int* vout, int n, int shift, const long long* offs, int nblk) {
  __shared__ long long base[256];
  __shared__ unsigned running[256];
  __shared__ unsigned wcnt[RS_THREADS / 32][256];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  base[t] = offs[(long long)t * nblk + blockIdx.x];
  running[t] = 0;
#pragma unroll
  for (int i = 0; i < RS_THREADS / 32; ++i) wcnt[i][t] = 0;
  __syncthreads();
  const unsigned lt_mask = (1u << lane) - 1u;
  long long tile = (long long)blockIdx.x * RS_TILE;
  for (int i = 0; i < RS_ITEMS; ++i) {
    long long idx = tile + (long long)i * RS_THREADS + t;
    bool valid = idx < n;
    unsigned long long key = valid ? kin[idx] : 0ull;
    int val = valid ? vin[idx] : 0;
    unsigned d = valid ? (unsigned)((key >> shift) & 255u) : 0xffffffffu;
    unsigned peers = __match_any_sync(SS_FULL_MASK, d);
    unsigned rank = __popc(peers & lt_mask);
    if (valid && rank == 0) wcnt[w][d] = __popc(peers);
    __syncthreads();
    if (valid) {
      unsigned before = running[d];
      for (int ww = 0; ww < w; ++ww) before += wcnt[ww][d];
      long long pos = base[d] + before + rank;
      kout[pos] = key;
      vout[pos] = val;
    }
    __syncthreads();
    unsigned add = 0;
#pragma unroll
    for (int ww = 0; ww < RS_THREADS / 32; ++ww) {
      add += wcnt[ww][t];
      wcnt[ww][t] = 0;
    }
    running[t] += add;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Builder kernels
// ---------------------------------------------------------------------------
__global__ void k_degrees(const long long* row_ptr, int n, int* deg, int* maxdeg) {
  int m = 0;
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    int d = (int)(row_ptr[v + 1] - row_ptr[v]);
    deg[v] = d;
    m = max(m, d);
  }
  m = __reduce_max_sync(SS_FULL_MASK, m);
  if ((threadIdx.x & 31) == 0) atomicMax(maxdeg, m);
}

__global__ void k_make_keys(const int* deg, int n, int sigma, int maxdeg, int dbits,
                            unsigned long long* keys, int* vals) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    unsigned long long win = (unsigned long long)(v / sigma);
    // a degree above maxdeg (possible only for inputs that break the caller's
    // contract) is clamped so that it cannot spill into the window bits
    keys[v] = (win << dbits) | (unsigned long long)(maxdeg - min(deg[v], maxdeg));
    vals[v] = (int)v;
  }
}

__global__ void k_identity(int* vals, int n) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x)
    vals[v] = (int)v;
}

// perm (padded), invperm, per-row degree; *n_live = 1 + the last row with a neighbour
__global__ void k_perm_tables(const int* sorted_vals, const int* deg, int n, int n_pad, int* perm,
                              int* invperm, int* rdeg, int* n_live) {
  int live = 0;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < n_pad;
       r += (long long)gridDim.x * blockDim.x) {
    if (r < n) {
      int v = sorted_vals[r];
      perm[r] = v;
      invperm[v] = (int)r;
      rdeg[r] = deg[v];
      if (deg[v] > 0) live = (int)r + 1;
    } else {
      perm[r] = -1;
      rdeg[r] = 0;
    }
  }
  live = __reduce_max_sync(SS_FULL_MASK, live);
  if ((threadIdx.x & 31) == 0 && live) atomicMax(n_live, live);
}

// cl[i] = longest row of chunk i; cs[i] = C * cl[i] (scanned afterwards); cs[n_c] = 0
// *busy = chunks with at least one column.
__global__ void k_chunk_len(const int* rdeg, int n_c, int C, int* cl, long long* cs, int* busy) {
  int mine = 0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i <= n_c;
       i += (long long)gridDim.x * blockDim.x) {
    if (i == n_c) {
      cs[i] = 0;
      continue;
    }
    int m = 0;
    for (int l = 0; l < C; ++l) m = max(m, rdeg[i * C + l]);
    cl[i] = m;
    cs[i] = (long long)C * m;
    mine += m > 0;
  }
  mine = __reduce_add_sync(SS_FULL_MASK, mine);
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(busy, mine);
}

// items per chunk for a given width W (0 = one item per chunk); split flags
__global__ void k_item_count(const int* cl, int n_c, int W, long long* cnt, long long* split_flag) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i <= n_c;
       i += (long long)gridDim.x * blockDim.x) {
    if (i == n_c) {
      cnt[i] = 0;
      if (split_flag) split_flag[i] = 0;
      continue;
    }
    int L = cl[i];
    bool split = (W > 0 && L > W);
    cnt[i] = (L == 0) ? 0 : (split ? (L + W - 1) / W : 1);  // chunks of isolated rows get no item
    if (split_flag) split_flag[i] = split ? 1 : 0;
  }
}

__global__ void k_item_fill(const int* cl, int n_c, int W, const long long* off,
                            const long long* split_idx, int4* items, int* split_n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_c;
       i += (long long)gridDim.x * blockDim.x) {
    int L = cl[i];
    long long o = off[i];
    if (W > 0 && L > W) {
      int cnt = (L + W - 1) / W;
      int s = split_idx ? (int)split_idx[i] : -1;
      for (int q = 0; q < cnt; ++q) items[o + q] = make_int4((int)i, q * W, min((q + 1) * W, L), s);
      if (split_n && s >= 0) split_n[s] = cnt;
    } else if (L > 0) {
      items[o] = make_int4((int)i, 0, L, -1);
    }
  }
}

// col[cs_i + j*C + l] for the columns of every item, one warp per item.  A lane owns a
// row (C = 64: two in turn; C < 32: 32 / C columns side by side) and walks its
// neighbours from the last, PACK_STEP at a time: consecutive entries of one row share
// sectors, and the stores of a column are coalesced.  Bound by the random gathers of
// invperm (one per edge, from L2); working out row and column of every slot anew, with
// four dependent loads each, took 2.2 ms on Kronecker 22; this one takes 0.86.
constexpr int PACK_STEP = 8;
template <int C>
__global__ void __launch_bounds__(256) k_pack(const int4* items, int n_items, const long long* cs,
                                              const int* perm, const int* __restrict__ invperm,
                                              const int* rdeg, const long long* row_ptr,
                                              const int* __restrict__ csr_col, int* __restrict__ col) {
  constexpr int ROWS = C < 32 ? C : 32, SIDE = 32 / ROWS;
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long it = wid; it < n_items; it += nw) {
    const int4 item = items[it];
    const long long c0 = cs[item.x];
#pragma unroll
    for (int l = lane % ROWS; l < C; l += 32) {
      const long long r = (long long)item.x * C + l;
      const int v = perm[r];
      const int deg = v >= 0 ? rdeg[r] : 0;
      const int* src = csr_col + (v >= 0 ? row_ptr[v + 1] - 1 : 0);
      int* dst = col + c0 + l;
      for (int j0 = item.y + lane / ROWS; j0 < item.z; j0 += PACK_STEP * SIDE) {
        int u[PACK_STEP];
#pragma unroll
        for (int q = 0; q < PACK_STEP; ++q) {
          const int j = j0 + q * SIDE;
          u[q] = (j < deg && j < item.z) ? __ldg(src - j) : -1;
        }
#pragma unroll
        for (int q = 0; q < PACK_STEP; ++q)
          if (u[q] >= 0) u[q] = __ldg(invperm + u[q]);
#pragma unroll
        for (int q = 0; q < PACK_STEP; ++q) {
          const int j = j0 + q * SIDE;
          if (j < item.z) dst[(long long)j * C] = u[q];
        }
      }
    }
  }
}

// Sort keys of the work items: longest first.
__global__ void k_item_keys(const int4* items, int n, int longest, unsigned long long* keys, int* vals) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    keys[i] = (unsigned long long)(longest - (items[i].z - items[i].y));
    vals[i] = (int)i;
  }
}

// Items by descending length (sorted) in snake order: position p of round p / W
// comes from the mirrored position in every other round.
__global__ void k_item_snake(const int4* items, const int* sorted, int n, int W, int4* out) {
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (long long)gridDim.x * blockDim.x) {
    const long long r = p / W, w = p % W, len = min((long long)W, n - r * W);
    out[p] = items[sorted[(r & 1) ? r * W + (len - 1 - w) : p]];
  }
}

static int bit_width(unsigned long long x) {
  int b = 0;
  while (x) {
    ++b;
    x >>= 1;
  }
  return b;
}

// Stable sort of n (key, value) pairs by the low `bits` bits; the sorted values end in *out.
static ss_status sort_pairs(unsigned long long* keys_a, unsigned long long* keys_b, int* vals_a, int* vals_b,
                            int n, int bits, long long* hist, long long* tmp_scan, int** out, cudaStream_t st) {
  const int nblk = (n + RS_TILE - 1) / RS_TILE;
  for (int shift = 0; shift < bits; shift += 8) {
    k_rs_hist<<<nblk, RS_THREADS, 0, st>>>(keys_a, n, shift, hist, nblk);
    ss_status s = excl_scan(hist, (long long)256 * nblk, tmp_scan, st);
    if (s != SS_OK) return s;
    k_rs_scatter<<<nblk, RS_THREADS, 0, st>>>(keys_a, vals_a, keys_b, vals_b, n, shift, hist, nblk);
    std::swap(keys_a, keys_b);
    std::swap(vals_a, vals_b);
  }
  SS_CUDA(cudaGetLastError());
  *out = vals_a;
  return SS_OK;
}

template <int C>
static void launch_pack(const slimsell_graph* h, const int4* items, int n_items, const long long* row_ptr,
                        const int* csr_col, cudaStream_t st) {
  k_pack<C><<<8 * h->num_sms, 256, 0, st>>>(items, n_items, h->cs, h->perm, h->invperm, h->rdeg, row_ptr,
                                            csr_col, h->col);
}

// Widest BFS items that the packing takes as they are (one warp each); wider ones
// (hub chunks unsplit) are packed from a table of their own.
constexpr int PACK_WIDTH = 1024;

// The layout's tables, but for the work items and columns.
static void add_tables(slimsell_graph* h, Slab& p) {
  const size_t np = (size_t)h->n_pad;
  p.add(&h->perm, np);
  p.add(&h->invperm, (size_t)h->n);
  p.add(&h->rdeg, np);
  p.add(&h->cl, (size_t)h->n_c);
  p.add(&h->cs, (size_t)h->n_c + 1);
}

// The BFS state whose size follows from n and nnz.
static void add_state(slimsell_graph* h, Slab& p) {
  const size_t np = (size_t)h->n_pad;
  // bitmap words rounded up to whole int4 groups, plus one spare group
  h->fb_words = (long long)((((np + 31) / 32) + 3) / 4 * 4 + 4);
  h->units_cap = (long long)np + h->nnz / 256 + 1024;  // any frontier fits
  h->iter_cap = 1 << 16;
  p.add(&h->claim, np);
  p.add(&h->vis, (size_t)h->fb_words);
  p.add(&h->act, (size_t)h->n_c);
  for (int b = 0; b < 2; ++b) p.add(&h->fb[b], (size_t)h->fb_words);
  p.add(&h->fr, np);
  p.add(&h->units, (size_t)h->units_cap);
  p.add(&h->psum, np);
  p.add(&h->touched, (size_t)h->fb_words);
  p.add(&h->qcount, 1);
  p.add(&h->ctl, 1);
  p.add(&h->feats, SS_SELECTOR_FEATURES * (size_t)h->iter_cap);
  p.add(&h->iters, (size_t)h->iter_cap);
  p.add(&h->lstat, SS_LSTAT * (size_t)h->iter_cap);
}

static ss_status clear_state(slimsell_graph* h, cudaStream_t st) {
  SS_CUDA(cudaMemsetAsync(h->psum, 0, sizeof(float) * (size_t)h->n_pad, st));
  SS_CUDA(cudaMemsetAsync(h->touched, 0, sizeof(unsigned) * (size_t)h->fb_words, st));
  SS_CUDA(cudaMemsetAsync(h->ctl, 0, sizeof(Ctl), st));
  return SS_OK;
}

// The state of a handle whose build had no room for it beside the temporaries.
static ss_status place_late_state(slimsell_graph* h, cudaStream_t st) {
  Slab p;
  add_state(h, p);
  ss_status s = p.place(h, &h->slab[2]);
  if (s == SS_OK) s = clear_state(h, st);
  if (s != SS_OK) return s;
  SS_CUDA(cudaStreamSynchronize(st));
  return SS_OK;
}

static ss_status build_impl(slimsell_graph* h, const long long* row_ptr, const int* csr_col, void** temps,
                            cudaStream_t st) {
  const int n = h->n, C = h->C;
  const int n_c = h->n_c, n_pad = h->n_pad;
  const int grid = 8 * h->num_sms;
  ss_status s;

  // temporaries (temps: allocations that the caller frees)
  int *deg = nullptr, *flags = nullptr, *vals_a = nullptr, *vals_b = nullptr;
  unsigned long long *keys_a = nullptr, *keys_b = nullptr;
  long long *hist = nullptr, *tmp_scan = nullptr, *cnt = nullptr, *split = nullptr, *pack_cnt = nullptr;
  const bool own_pack = h->split_w <= 0 || h->split_w > PACK_WIDTH;
  const int nblk = (n + RS_TILE - 1) / RS_TILE;
  const long long scan_len = std::max<long long>((long long)256 * nblk, (long long)n_c + 1);
  {
    Slab t;
    t.add(&deg, (size_t)n);
    t.add(&flags, 3);  // largest degree, live rows, busy chunks
    t.add(&vals_a, (size_t)n);
    t.add(&vals_b, (size_t)n);
    t.add(&keys_a, (size_t)n);
    t.add(&keys_b, (size_t)n);
    t.add(&hist, (size_t)256 * nblk);
    t.add(&tmp_scan, (size_t)(scan_len / SCAN_TILE + 2));
    t.add(&cnt, (size_t)n_c + 1);
    t.add(&split, (size_t)n_c + 1);
    if (own_pack) t.add(&pack_cnt, (size_t)n_c + 1);
    if ((s = t.place(nullptr, &temps[0])) != SS_OK) return s;
  }

  // permanent arrays whose size follows from n and nnz: the layout's tables and the BFS state,
  // which waits for the temporaries to be gone where the device does not hold both
  {
    Slab p;
    add_tables(h, p);
    add_state(h, p);
    s = p.place(h, &h->slab[0]);
    if (s == SS_OK) {
      if ((s = clear_state(h, st)) != SS_OK) return s;
    } else if (s == SS_ERR_OOM) {
      set_error("");
      h->claim = nullptr;
      Slab q;
      add_tables(h, q);
      s = q.place(h, &h->slab[0]);
    }
    if (s != SS_OK) return s;
  }

  // 1. degrees and sort keys
  SS_CUDA(cudaMemsetAsync(flags, 0, 3 * sizeof(int), st));
  k_degrees<<<grid, 256, 0, st>>>(row_ptr, n, deg, flags);
  SS_CUDA(cudaMemcpyAsync(&h->max_degree, flags, sizeof(int), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));

  // 2. sigma-window sort by descending degree (stable: ties keep ascending id)
  int* sorted = vals_a;
  if (h->sigma <= 1) {
    k_identity<<<grid, 256, 0, st>>>(vals_a, n);
  } else {
    const int sigma = h->sigma >= n ? n : h->sigma;  // already a multiple of C (or >= n)
    const int dbits = bit_width((unsigned long long)h->max_degree);
    const long long nwin = ((long long)n + sigma - 1) / sigma;
    const int bits = dbits + bit_width((unsigned long long)(nwin - 1));
    k_make_keys<<<grid, 256, 0, st>>>(deg, n, sigma, h->max_degree, dbits, keys_a, vals_a);
    if ((s = sort_pairs(keys_a, keys_b, vals_a, vals_b, n, bits, hist, tmp_scan, &sorted, st)) != SS_OK) return s;
  }
  SS_CUDA(cudaGetLastError());

  // 3. perm / invperm / row degrees, chunk lengths and starts, work items per chunk
  k_perm_tables<<<grid, 256, 0, st>>>(sorted, deg, n, n_pad, h->perm, h->invperm, h->rdeg, flags + 1);
  k_chunk_len<<<grid, 256, 0, st>>>(h->rdeg, n_c, C, h->cl, h->cs, flags + 2);
  k_item_count<<<grid, 256, 0, st>>>(h->cl, n_c, h->split_w, cnt, split);
  if (own_pack) k_item_count<<<grid, 256, 0, st>>>(h->cl, n_c, 256, pack_cnt, nullptr);
  SS_CUDA(cudaGetLastError());
  if ((s = excl_scan(h->cs, n_c + 1, tmp_scan, st)) != SS_OK) return s;
  if ((s = excl_scan(cnt, n_c + 1, tmp_scan, st)) != SS_OK) return s;
  if ((s = excl_scan(split, n_c + 1, tmp_scan, st)) != SS_OK) return s;
  if (own_pack && (s = excl_scan(pack_cnt, n_c + 1, tmp_scan, st)) != SS_OK) return s;
  long long slots = 0, nitems = 0, nsplit = 0, npack = 0;
  SS_CUDA(cudaMemcpyAsync(&slots, h->cs + n_c, sizeof(long long), cudaMemcpyDeviceToHost, st));
  int rows_chunks[2] = {0, 0};
  SS_CUDA(cudaMemcpyAsync(rows_chunks, flags + 1, 2 * sizeof(int), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaMemcpyAsync(&nitems, cnt + n_c, sizeof(long long), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaMemcpyAsync(&nsplit, split + n_c, sizeof(long long), cudaMemcpyDeviceToHost, st));
  if (own_pack) SS_CUDA(cudaMemcpyAsync(&npack, pack_cnt + n_c, sizeof(long long), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  if (nitems > 0x7fffffffLL || npack > 0x7fffffffLL) {
    set_error("too many work items (%lld)", std::max(nitems, npack));
    return SS_ERR_UNSUPPORTED;
  }
  h->n_live = rows_chunks[0];
  h->n_busy = rows_chunks[1];
  h->slots = slots;
  h->n_items = (int)nitems;
  h->n_split = (int)nsplit;

  // permanent arrays whose size follows from the layout; temporaries of the item order
  // block units cover PUSH_BLOCK_SLOTS / C columns each: at most one partial unit per chunk
  h->bunits_cap = (long long)n_c + slots / PUSH_BLOCK_SLOTS + 1024;
  {
    Slab p;
    p.add(&h->col, (size_t)slots);
    p.add(&h->items, (size_t)nitems);
    p.add(&h->split_n, (size_t)nsplit);
    p.add(&h->xacc, (size_t)nsplit * C);
    p.add(&h->xpar, (size_t)nsplit * C);
    p.add(&h->arrive, (size_t)nsplit);
    p.add(&h->bunits, (size_t)h->bunits_cap);
    if ((s = p.place(h, &h->slab[1])) != SS_OK) return s;
  }
  SS_CUDA(cudaMemsetAsync(h->arrive, 0, sizeof(unsigned) * (size_t)std::max(nsplit, 1LL), st));
  int4 *fresh = nullptr, *pack_items = nullptr;
  unsigned long long *ik_a = keys_a, *ik_b = keys_b;
  int *iv_a = vals_a, *iv_b = vals_b;
  long long *ihist = hist, *iscan = tmp_scan;
  {
    const size_t iblk = (size_t)((nitems + RS_TILE - 1) / RS_TILE);
    Slab t;
    t.add(&fresh, (size_t)nitems);
    if (own_pack) t.add(&pack_items, (size_t)npack);
    if (nitems > n) {  // (narrow splits: more items than vertices)
      t.add(&ik_a, (size_t)nitems);
      t.add(&ik_b, (size_t)nitems);
      t.add(&iv_a, (size_t)nitems);
      t.add(&iv_b, (size_t)nitems);
      t.add(&ihist, 256 * iblk);
      t.add(&iscan, 256 * iblk / SCAN_TILE + 2);
    }
    if ((s = t.place(nullptr, &temps[1])) != SS_OK) return s;
  }

  // 4. the BFS work items, ordered for the iteration kernels, whose warp w takes items
  // w, w + W, w + 2W, ... (W = warps in the grid): longest first, and every other group of
  // W items is reversed ("snake" order) so each warp's total is balanced
  k_item_fill<<<grid, 256, 0, st>>>(h->cl, n_c, h->split_w, cnt, split, fresh, h->split_n);
  if (nitems > 0) {
    const int longest = h->split_w > 0 ? std::min(h->split_w, h->max_degree) : h->max_degree;
    int* order = nullptr;
    k_item_keys<<<grid, 256, 0, st>>>(fresh, h->n_items, longest, ik_a, iv_a);
    if ((s = sort_pairs(ik_a, ik_b, iv_a, iv_b, h->n_items, bit_width((unsigned long long)(longest - 1)), ihist,
                        iscan, &order, st)) != SS_OK)
      return s;
    k_item_snake<<<grid, 256, 0, st>>>(fresh, order, h->n_items, h->num_sms * (SS_PULL_THREADS / 32), h->items);
  }
  if (own_pack) k_item_fill<<<grid, 256, 0, st>>>(h->cl, n_c, 256, pack_cnt, nullptr, pack_items, nullptr);
  SS_CUDA(cudaGetLastError());

  // 5. pack
  const int4* pitems = own_pack ? pack_items : h->items;
  const int np_items = own_pack ? (int)npack : h->n_items;
  switch (C) {
    case 8: launch_pack<8>(h, pitems, np_items, row_ptr, csr_col, st); break;
    case 16: launch_pack<16>(h, pitems, np_items, row_ptr, csr_col, st); break;
    case 32: launch_pack<32>(h, pitems, np_items, row_ptr, csr_col, st); break;
    default: launch_pack<64>(h, pitems, np_items, row_ptr, csr_col, st); break;
  }
  SS_CUDA(cudaGetLastError());
  SS_CUDA(cudaStreamSynchronize(st));
  return SS_OK;
}

// Host-side state of a handle.
static ss_status host_state(slimsell_graph* h) {
  h->local_cluster = push_local_cluster_size();
  if (h->local_cluster <= 0) {
    set_error("slimsell_build: no thread-block cluster of the push kernel fits on this device");
    return SS_ERR_CUDA;
  }
  SS_CUDA(cudaHostAlloc((void**)&h->h_ctl, sizeof(Ctl), cudaHostAllocDefault));
  SS_CUDA(cudaEventCreate(&h->ev_a));
  SS_CUDA(cudaEventCreate(&h->ev_b));
  SS_CUDA(cudaEventCreate(&h->ev_c));
  SS_CUDA(cudaEventCreate(&h->ev_d));
  SS_CUDA(cudaEventCreateWithFlags(&h->ev_done, cudaEventDisableTiming));
  return SS_OK;
}

void ab_release(slimsell_graph* h);  // format-comparison scratch (ss_sell.cu)
void bc_release(slimsell_graph* h);  // betweenness-centrality scratch (ss_bc.cu)

void free_handle(slimsell_graph* h) {
  if (!h) return;
  ab_release(h);
  bc_release(h);
  void* ptrs[] = {h->slab[0], h->slab[1], h->slab[2], h->mlp, h->mF[0], h->mF[1], h->mV, h->mxacc, h->mroots, h->mplanes[0], h->mplanes[1]};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (h->h_ctl) cudaFreeHost(h->h_ctl);
  if (h->ev_a) cudaEventDestroy(h->ev_a);
  if (h->ev_b) cudaEventDestroy(h->ev_b);
  if (h->ev_c) cudaEventDestroy(h->ev_c);
  if (h->ev_d) cudaEventDestroy(h->ev_d);
  for (cudaEvent_t e : h->evq) cudaEventDestroy(e);
  if (h->ev_done) {
    cudaEventSynchronize(h->ev_done);
    cudaEventDestroy(h->ev_done);
  }
  for (auto& row : h->loop_exec)
    for (auto& e : row)
      if (e) cudaGraphExecDestroy(e);
  delete h;
}

}  // namespace ss

ss::Dev slimsell_graph::dev() const {
  ss::Dev d;
  d.n = n; d.C = C; d.n_c = n_c; d.n_pad = n_pad; d.n_items = n_items; d.n_split = n_split;
  d.perm = perm; d.invperm = invperm; d.rdeg = rdeg; d.cl = cl; d.cs = cs; d.col = col;
  d.items = items; d.split_n = split_n; d.claim = claim; d.vis = vis; d.act = act;
  d.n_live = n_live; d.max_degree = max_degree; d.n_busy = n_busy;
  d.fb[0] = fb[0]; d.fb[1] = fb[1]; d.fb_words = fb_words;
  // staged prefix: whole int4 groups, never past the allocated bitmap
  long long need = ((((long long)n_pad + 31) / 32) + 3) / 4 * 4;
  long long cap = (long long)(smem_bytes / 16) * 4;
  d.smem_words = (int)(need < cap ? need : cap);
  d.fr = fr; d.xacc = xacc; d.xpar = xpar; d.arrive = arrive;
  d.units = units; d.units_cap = units_cap;
  d.bunits = bunits; d.bunits_cap = bunits_cap; d.push_blocks = push_blocks;
  d.format = SS_FORMAT_SLIMSELL; d.scol = nullptr; d.sval = nullptr;  // set per call by slimsell_bfs
  d.psum = psum; d.touched = touched; d.mlp = mlp; d.feats = feats;
  d.sel_margin = sel_margin;
  d.qcount = qcount;
  d.local_cluster = local_cluster;
  d.local_max_nf = (long long)local_cluster * SS_LOCAL_SLICE;
  d.local_max_e = (long long)local_cluster * SS_LOCAL_EDGES_PER_CTA;
  d.nnz = nnz; d.total_slots = slots; d.reach_cap = (unsigned long long)n;
  d.ctl = ctl; d.iters = iters; d.iter_cap = iter_cap; d.lstat = lstat;
  return d;
}

extern "C" {

ss_status slimsell_build(const int64_t* d_row_ptr, const int32_t* d_col, int32_t n, int64_t nnz,
                         int32_t C, int32_t sigma, int32_t split_w, void* stream,
                         slimsell_handle* out) {
  ss::set_error("");
  if (!out) {
    ss::set_error("slimsell_build: out is NULL");
    return SS_ERR_INVALID;
  }
  *out = nullptr;
  if (n < 1 || nnz < 0 || !d_row_ptr || (nnz > 0 && !d_col)) {
    ss::set_error("slimsell_build: bad graph arguments (n=%d nnz=%lld)", n, (long long)nnz);
    return SS_ERR_INVALID;
  }
  if (!(C == 8 || C == 16 || C == 32 || C == 64)) {
    ss::set_error("slimsell_build: C must be 8, 16, 32 or 64 (got %d)", C);
    return SS_ERR_INVALID;
  }
  if (sigma < 1 || split_w < 0) {
    ss::set_error("slimsell_build: sigma must be >= 1 and split_w >= 0");
    return SS_ERR_INVALID;
  }
  long long n_c = ((long long)n + C - 1) / C;
  if (n_c * C > 0x7fffffffLL) {
    ss::set_error("slimsell_build: n too large for int32 row ids");
    return SS_ERR_UNSUPPORTED;
  }
  slimsell_graph* h = new slimsell_graph();
  cudaStream_t st = (cudaStream_t)stream;
  cudaGetDevice(&h->device);
  cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, h->device);
  h->n = n;
  h->nnz = nnz;
  h->C = C;
  // sigma > 1 is rounded up to a multiple of C (the paper takes it as one, Section IV)
  h->sigma = sigma <= 1 ? 1 : (int)std::min<long long>(((long long)sigma + C - 1) / C * C, INT_MAX);
  h->split_w = split_w;
  h->n_c = (int)n_c;
  h->n_pad = (int)(n_c * C);
  void* temps[2] = {nullptr, nullptr};
  ss_status s = ss::host_state(h);
  if (s == SS_OK) s = ss::build_impl(h, (const long long*)d_row_ptr, d_col, temps, st);
  if (s != SS_OK) cudaStreamSynchronize(st);  // queued work may still use the temporaries
  for (void* t : temps)
    if (t) cudaFree(t);
  if (s == SS_OK && !h->claim) s = ss::place_late_state(h, st);
  if (s != SS_OK) {
    ss::free_handle(h);
    return s;
  }
  *out = h;
  return SS_OK;
}

const char* slimsell_last_error(void) { return ss::last_error(); }

const char* slimsell_version(void) { return "slimsell-gb300 0.1 (sm_103a)"; }

void slimsell_destroy(slimsell_handle h) { ss::free_handle(h); }

ss_status slimsell_get_info(slimsell_handle h, ss_info* out) {
  if (!h || !out) {
    ss::set_error("slimsell_get_info: NULL argument");
    return SS_ERR_INVALID;
  }
  out->n = h->n; out->C = h->C; out->sigma = h->sigma; out->split_w = h->split_w;
  out->n_chunks = h->n_c; out->n_items = h->n_items; out->n_split_chunks = h->n_split;
  out->max_degree = h->max_degree; out->nnz = h->nnz; out->slots = h->slots;
  out->padding = h->slots - h->nnz; out->device_bytes = h->device_bytes;
  return SS_OK;
}

ss_status slimsell_export_layout(slimsell_handle h, int32_t* d_perm, int32_t* d_cl, int64_t* d_cs,
                                 int32_t* d_col, int32_t* d_items, void* stream) {
  if (!h) {
    ss::set_error("slimsell_export_layout: NULL handle");
    return SS_ERR_INVALID;
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (d_perm) SS_CUDA(cudaMemcpyAsync(d_perm, h->perm, sizeof(int) * (size_t)h->n_pad, cudaMemcpyDeviceToDevice, st));
  if (d_cl) SS_CUDA(cudaMemcpyAsync(d_cl, h->cl, sizeof(int) * (size_t)h->n_c, cudaMemcpyDeviceToDevice, st));
  if (d_cs) SS_CUDA(cudaMemcpyAsync(d_cs, h->cs, sizeof(long long) * (size_t)(h->n_c + 1), cudaMemcpyDeviceToDevice, st));
  if (d_col && h->slots > 0) SS_CUDA(cudaMemcpyAsync(d_col, h->col, sizeof(int) * (size_t)h->slots, cudaMemcpyDeviceToDevice, st));
  if (d_items && h->n_items > 0) SS_CUDA(cudaMemcpyAsync(d_items, h->items, sizeof(int4) * (size_t)h->n_items, cudaMemcpyDeviceToDevice, st));
  SS_CUDA(cudaStreamSynchronize(st));
  return SS_OK;
}

}  // extern "C"
