// Multi-source BFS: the boolean semiring of Section III-A run for up to 1024
// sources at once with bit-packed frontiers (an extension beyond the paper).
//
//   F[k&1][r][w]  bit s of word w: row r entered source 64w+s's frontier at level k
//   V[r][w]       visited bits (g_k = not V)
//   x = OR over the row's neighbours u of F[u][w]; new = x & ~V; V |= new;
//   F_next = new; dist[v][64w+s] = k for every new bit.
//
// One thread block handles one work item (chunk i, columns [j0, j1)); thread
// (r, w) = threadIdx.x / W, % W owns word w of row r.  The W threads of a row
// read the same col entry (a broadcast) and gather the W contiguous frontier
// words of the neighbour (one W*8-byte segment).  SlimWork skips chunks whose
// rows have every source visited; split chunks (SlimChunk) combine partial ORs
// with 64-bit atomicOr and the last arriving block post-processes.
//
// The gathers are most of the traffic (W*8 bytes per slot), so they are
// skipped where they cannot matter: a one-bit-per-vertex summary of the
// frontier (bit u set iff some source has u in its frontier, kept in the
// single-source frontier bitmaps fb[], unused here) is tested first, and a
// thread whose 64 sources have all visited its row gathers nothing.
//
// Parents (optional) come from a separate pass after each level: a row's
// neighbours are stored in descending original id, so for each source that
// the row gained at level k, the first neighbour in storage order that was in
// that source's level-(k-1) frontier is its largest-id parent.  The pass
// reads F[(k-1)&1] and the summary bitmap of level k-1, both still intact
// until level k+1 overwrites them.
#include <algorithm>
#include <cstdint>
#include <vector>

#include "ss_pull.cuh"

namespace ss {

#ifndef SS_MULTI_BATCH
#define SS_MULTI_BATCH 4
#endif
constexpr int MULTI_BATCH = SS_MULTI_BATCH;  // columns per thread in flight
#ifndef SS_MULTI_BLOCKS_PER_SM
#define SS_MULTI_BLOCKS_PER_SM 0  // resident blocks per SM (0: as many as fit)
#endif

// Levels are kept as bit planes until the end of an epoch of 2^P - 1 levels: the P
// planes of word (row, w) hold the bits of the level (within the epoch) at which the row
// entered each of the 64 sources' frontiers.  k_multi_levels then writes the distances in
// vertex order.  Written at each discovery instead, into an array first filled with -1, they
// were 16-byte read-modify-writes scattered over the n x k output: 0.8 of the 2.5 ms of
// 64 sources on Kronecker 22 (0.64 in the pulls, 0.16 the fill).
// The first epoch has four planes, a 32-byte sector a word, which most runs end in.  A longer
// run goes on with eight in an array of their own, 255 levels an epoch: an epoch's end (the
// writes, and the planes cleared) is 22 us on a 512^2 lattice, 3 to 4 % of a run of a thousand
// levels that paid it every 15.  Where their memory is not to be had the epochs stay short.
constexpr int MULTI_SHORT_PLANES = 4, MULTI_LONG_PLANES = 8;
constexpr int MULTI_EPOCH = (1 << MULTI_SHORT_PLANES) - 1, MULTI_EPOCH_LONG = (1 << MULTI_LONG_PLANES) - 1;

// How a level pass keeps its levels: not (written at once, or not wanted), in the planes of the
// short first epoch, or in those of a long one.  A parameter of the kernels, each form with
// its own code, as the gather loops' register allocation follows the slightest change of it.
enum { KEEP_NOT = 0, KEEP_SHORT = 1, KEEP_LONG = 2 };
template <int KEEP>
__host__ __device__ constexpr int planes_of() { return KEEP == KEEP_LONG ? MULTI_LONG_PLANES : MULTI_SHORT_PLANES; }

// Out of line, so that the gather loops' register allocation does not depend on it.
template <int KEEP>
__device__ __noinline__ void keep_levels(unsigned long long* planes, unsigned long long nb, int level) {
  const int code = KEEP == KEEP_LONG ? (level - 1 - MULTI_EPOCH) % MULTI_EPOCH_LONG + 1 : (level - 1) % MULTI_EPOCH + 1;
#pragma unroll
  for (int i = 0; i < planes_of<KEEP>(); ++i)
    if (code >> i & 1) planes[i] |= nb;
}

// The other way, at each discovery into an output first filled with -1, stays for
// outputs of fewer than MULTI_PLANES_OUT entries, where k_multi_levels' launch and latency
// are not made up for (32 sources on Kronecker 16: 376 us; by way of planes 408), and
// for k of at most half the words' sources, whose planes are mostly empty (48 sources in
// two words on Kronecker 20: 1115 us and 1188; 2 on Kronecker 21, with parents: 1.34 ms
// and 1.89).  Also where the planes do not fit in the device's memory.
constexpr long long MULTI_PLANES_OUT = 16LL << 20;
static bool multi_planes(const slimsell_graph* h, int k, int W) {
  return k > 32 * W && (long long)h->n * k >= MULTI_PLANES_OUT;
}

// Distances of the new sources (bits of nb) of one 64-source word, in 16-byte
// groups of 4: a group with no earlier discovery (bits of vold) still holds -1
// everywhere and is written whole; otherwise it is read first.  Kept out of line
// so that the gather loop's register allocation does not depend on it.
__device__ __noinline__ void write_levels_vec(int* out, unsigned long long nb, unsigned long long vold,
                                             int level) {
  for (int gi = 0; gi < 16; ++gi) {
    const unsigned ng = (unsigned)(nb >> (4 * gi)) & 0xFu;
    if (!ng) continue;
    int4* q = reinterpret_cast<int4*>(out) + gi;
    int4 v = ((unsigned)(vold >> (4 * gi)) & 0xFu) ? *q : make_int4(-1, -1, -1, -1);
    if (ng & 1u) v.x = level;
    if (ng & 2u) v.y = level;
    if (ng & 4u) v.z = level;
    if (ng & 8u) v.w = level;
    *q = v;
  }
}

// Distances of an epoch (levels base + 1 on) from its P planes; the
// first epoch writes every entry (-1 where nothing was found), later ones what they
// found, and the planes are cleared for the next.  Sixteen lanes write the 64
// entries of a vertex's word as 16-byte groups where the output allows it.  (In row
// order the writes of 256 bytes went to scattered places: 347 us on Kronecker 22.)
template <int P>
__global__ void __launch_bounds__(256) k_multi_levels(MultiDev m, int W, int lgW, int base) {
  const Dev& d = m.d;
  const long long words = (long long)d.n << lgW;  // word i: word i & (W - 1) of vertex i >> lgW
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long groups = (long long)gridDim.x * blockDim.x >> 4;  // 16 lanes each
  const int g = (int)(t & 15);
  constexpr int U = 16 / P;  // words in flight per group
  for (long long w0 = t >> 4; w0 < words; w0 += U * groups) {
    unsigned b[U][P], found[U];
    int row[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long word = w0 + u * groups;
      row[u] = word < words ? __ldg(d.invperm + (word >> lgW)) : d.n_live;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      found[u] = 0;
#pragma unroll
      for (int p = 0; p < P; ++p) b[u][p] = 0;
      if (row[u] < d.n_live) {  // (rows without neighbours have no levels)
        const ulonglong2* q = reinterpret_cast<const ulonglong2*>(
            m.planes + (((long long)row[u] << lgW) + ((w0 + u * groups) & (W - 1))) * P);
#pragma unroll
        for (int p = 0; p < P; p += 2) {
          const ulonglong2 x = __ldg(q + p / 2);
          b[u][p] = (unsigned)(x.x >> (4 * g)) & 0xFu;
          b[u][p + 1] = (unsigned)(x.y >> (4 * g)) & 0xFu;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long word = w0 + u * groups;
      const int s0 = 64 * (int)(word & (W - 1)) + 4 * g;
#pragma unroll
      for (int p = 0; p < P; ++p) found[u] |= b[u][p];
      if (word >= words || s0 >= m.k || (base > 0 && !found[u])) continue;
      int v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        int code = 0;
#pragma unroll
        for (int p = 0; p < P; ++p) code |= (b[u][p] >> j & 1u) << p;
        v[j] = code ? base + code : -1;
      }
      int* out = m.dist + (word >> lgW) * m.k + s0;
      if (m.vec_dist && (base == 0 || found[u] == 0xFu)) {
        __stcs(reinterpret_cast<int4*>(out), make_int4(v[0], v[1], v[2], v[3]));
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (s0 + j < m.k && (base == 0 || v[j] >= 0)) out[j] = v[j];
      }
    }
  }
}

// The sources' own distances, after the first epoch has written every entry.
__global__ void k_multi_root_levels(MultiDev m) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < m.k; s += gridDim.x * blockDim.x)
    m.dist[(long long)m.roots[s] * m.k + s] = 0;
}

// Resident blocks asked of the compiler (0: its choice) so that MULTI_BATCH columns stay in
// flight: left alone, it gave the plane form of some shapes fewer registers than the loads
// take and a spill (64 sources in chunks of 64: 32 registers; Kronecker 20 in items of 1024
// columns 2407 us, 1247 with 40; 128 sources there 1869 us, 1504 with 64).  Two words in chunks
// of 32 are worth 48: with 40 and a spill 100 sources on Kronecker 20 take 1029 us against
// 1084, but 128 on a 512^2 lattice 39.3 ms against 36.1.
template <int C, int W, int KEEP>
__host__ __device__ constexpr int multi_blocks() {
  if (KEEP == KEEP_NOT) return 0;
  if (C == 64 && W == 2) return 8;
  if (C == 32 && W == 2) return 20;
  return C * W == 64 ? 24 : 0;
}

template <int C, int W, bool SLIMWORK, int KEEP>
__global__ void __launch_bounds__(C * W, multi_blocks<C, W, KEEP>()) k_multi_pull(MultiDev m, IterLaunch il) {
  constexpr int T = C * W;
  const Dev& d = m.d;
  Ctl* c = d.ctl;
  if (c->done) return;
  const int level = c->k;
  const int tid = threadIdx.x, r = tid / W, w = tid % W;
  const unsigned long long* Fp = m.F[(level - 1) & 1];
  unsigned long long* Fn = m.F[level & 1];
  const unsigned* FAp = d.fb[(level - 1) & 1];  // frontier summary, one bit per row
  unsigned* FAn = d.fb[level & 1];
  __shared__ int s_flag;
  __shared__ unsigned s_fa[2];
  unsigned long long nw = 0, deg = 0, slots = 0, act = 0;
  unsigned maxdeg = 0;
  __shared__ unsigned long long s_rowdeg;  // degree sum of the block's rows that gained a source
  if (tid == 0) s_rowdeg = 0ull;
  for (int it = blockIdx.x; it < d.n_items; it += gridDim.x) {
    const int4 item = d.items[it];
    const int chunk = item.x;
    const long long row = (long long)chunk * C + r;
    if (SLIMWORK) {
      const int a = d.act[chunk];
      __syncthreads();  // every thread has read the state before it may change
      if (a != 1) {
        if (a >= 2 && item.y == 0) {
          Fn[row * W + w] = 0ull;  // f_k is zero on a finished chunk
          if (tid == 0) {
            store_bits<C>(FAn, chunk, 0u, 0u);
            d.act[chunk] = (a == 3) ? 2 : 0;
          }
        }
        continue;
      }
    }
    const long long start = d.cs[chunk] + (long long)item.y * C;
    const int ncol = item.z - item.y;
    const unsigned long long vold0 = m.V[row * W + w];
    const bool want = vold0 != ~0ull;  // some of this word's sources still miss the row
    unsigned long long acc = 0ull;
    int j = 0;
    for (; j + MULTI_BATCH <= ncol; j += MULTI_BATCH) {
      int cc[MULTI_BATCH];
#pragma unroll
      for (int q = 0; q < MULTI_BATCH; ++q) cc[q] = __ldcs(d.col + start + (long long)(j + q) * C + r);
      unsigned hit[MULTI_BATCH];
#pragma unroll
      for (int q = 0; q < MULTI_BATCH; ++q)
        hit[q] = (want && cc[q] >= 0) ? (__ldg(FAp + (cc[q] >> 5)) >> (cc[q] & 31)) & 1u : 0u;
#pragma unroll
      for (int q = 0; q < MULTI_BATCH; ++q)
        if (hit[q]) acc |= __ldg(Fp + (long long)cc[q] * W + w);
    }
    for (; j < ncol; ++j) {
      const int cc = __ldcs(d.col + start + (long long)j * C + r);
      if (want && cc >= 0 && ((__ldg(FAp + (cc >> 5)) >> (cc & 31)) & 1u))
        acc |= __ldg(Fp + (long long)cc * W + w);
    }
    if (tid == 0) slots += (unsigned long long)ncol * C;
    if (item.w >= 0) {  // SlimChunk: OR the partial rows, last block to arrive post-processes
      unsigned long long* xa = m.xacc + ((size_t)item.w * C + r) * W + w;
      if (acc) atomicOr(xa, acc);
      __threadfence();
      __syncthreads();
      if (tid == 0) {
        const unsigned old = atomicAdd(d.arrive + item.w, 1u);
        s_flag = (old == (unsigned)d.split_n[item.w] - 1u);
      }
      __syncthreads();
      if (!s_flag) continue;
      __threadfence();
      acc = __ldcg(xa);
      *xa = 0ull;
      if (tid == 0) d.arrive[item.w] = 0u;
    }
    if (tid == 0) s_fa[0] = s_fa[1] = 0u;
    __syncthreads();
    const unsigned long long vold = vold0;
    const unsigned long long nb = acc & ~vold;
    if (nb) atomicOr(&s_fa[r >> 5], 1u << (r & 31));
    if (nb) {
      m.V[row * W + w] = vold | nb;
      const int pc = __popcll(nb);
      const int dv = d.rdeg[row];
      nw += (unsigned long long)pc;
      deg += (unsigned long long)pc * (unsigned long long)dv;
      maxdeg = max(maxdeg, (unsigned)dv);
      if constexpr (KEEP != KEEP_NOT) {
        keep_levels<KEEP>(m.planes + (row * W + w) * planes_of<KEEP>(), nb, level);
      } else if (m.dist) {
        int* out = m.dist + (long long)d.perm[row] * m.k + 64 * w;
        if (m.vec_dist) {
          write_levels_vec(out, nb, vold, level);
        } else {
          unsigned long long b = nb;
          while (b) {
            const int s = __ffsll((long long)b) - 1;
            b &= b - 1;
            out[s] = level;
          }
        }
      }
    }
    Fn[row * W + w] = nb;
    const int left = __syncthreads_or((vold | nb) != ~0ull);
    if (w == 0 && ((s_fa[r >> 5] >> (r & 31)) & 1u)) atomicAdd(&s_rowdeg, (unsigned long long)d.rdeg[row]);
    if (tid == 0) {
      store_bits<C>(FAn, chunk, s_fa[0], s_fa[1]);
      d.act[chunk] = left ? 1 : 3;
      act += 1;
    }
  }
  // degree sum of the rows that gained a source, each row counted once (the
  // parents pass picks its direction from it)
  __syncthreads();
  if (tid == 0 && s_rowdeg) {
    atomicAdd(&c->new_rowdeg, s_rowdeg);
    __threadfence();  // before this block counts itself done
  }
  finish_iteration_block<T>(d, nw, deg, slots, act, maxdeg, il);
}

// The level pull for one word of sources (k <= 64): as k_multi_pull, with the pull
// kernel's layout.  One persistent block per SM stages the frontier summary's prefix
// in shared memory; a warp takes an item (chunks of at most MULTI_SHORT columns go
// 32 / Q at a time), lane l loading 16-byte quads of col and keeping the words of
// rows 4 (l mod Q) .. + 3.  A thread per row read the summary and the words from
// global memory, two dependent gathers a slot, 32 one-warp blocks an SM; here the
// summary bit is a shared-memory lookup, and a word is gathered (8 bytes, mostly from
// L2) only where some source has the neighbour in its frontier and some source
// still misses the row.  64 sources on Kronecker 22: the first two levels 283 and 376 us in
// k_multi_pull, 185 and 272 here.
#ifndef SS_MULTI_ONE_THREADS
#define SS_MULTI_ONE_THREADS 640
#endif
#ifndef SS_MULTI_ONE_STEP
#define SS_MULTI_ONE_STEP 4
#endif
constexpr int MULTI_ONE_THREADS = SS_MULTI_ONE_THREADS;
constexpr int MULTI_ONE_STEP = SS_MULTI_ONE_STEP;  // quads in flight per lane
constexpr int MULTI_SHORT = 4;

struct OneSum {
  unsigned long long nw = 0, deg = 0, rowdeg = 0;
  unsigned quads = 0, act = 0, maxdeg = 0;
};

// OR the frontier words of U quads into the rows' accumulators: every summary lookup
// of the step first, then every gather.
template <int U>
__device__ __forceinline__ void one_step(const unsigned* sm, int sbits, const unsigned* FAp,
                                         const unsigned long long* Fp, const int4* c, unsigned live,
                                         unsigned long long acc[4]) {
  unsigned hit = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int cc[4] = {c[u].x, c[u].y, c[u].z, c[u].w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
      hit |= frontier_bit(sm, sbits, FAp, (live >> r & 1u) ? cc[r] : -1) << (4 * u + r);
  }
  if (!hit) return;
  unsigned long long f[U][4];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int cc[4] = {c[u].x, c[u].y, c[u].z, c[u].w};
#pragma unroll
    for (int r = 0; r < 4; ++r) f[u][r] = (hit >> (4 * u + r) & 1u) ? __ldg(Fp + cc[r]) : 0ull;
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r] |= f[u][r];
}

// New words of four rows (from R0): visited and frontier words, level planes,
// counters; returns the bits of the rows that gained a source, *left = some row
// still misses one.
template <int KEEP>
__device__ __forceinline__ unsigned one_post(const MultiDev& m, long long R0, int level,
                                             const unsigned long long acc[4], const unsigned long long V[4],
                                             unsigned long long* Fn, OneSum& sum, bool* left) {
  const Dev& d = m.d;
  unsigned long long nb[4];
  unsigned nib = 0;
  *left = false;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    nb[r] = acc[r] & ~V[r];
    if (nb[r]) nib |= 1u << r;
    if ((V[r] | nb[r]) != ~0ull) *left = true;
  }
  ulonglong2* fn = reinterpret_cast<ulonglong2*>(Fn + R0);
  fn[0] = make_ulonglong2(nb[0], nb[1]);
  fn[1] = make_ulonglong2(nb[2], nb[3]);
  if (nib) {
    ulonglong2* vv = reinterpret_cast<ulonglong2*>(m.V + R0);
    vv[0] = make_ulonglong2(V[0] | nb[0], V[1] | nb[1]);
    vv[1] = make_ulonglong2(V[2] | nb[2], V[3] | nb[3]);
    const int4 dg = *reinterpret_cast<const int4*>(d.rdeg + R0);
    const int D[4] = {dg.x, dg.y, dg.z, dg.w};
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (nib >> r & 1u) {
        const int pc = __popcll(nb[r]);
        sum.nw += (unsigned long long)pc;
        sum.deg += (unsigned long long)pc * (unsigned long long)D[r];
        sum.rowdeg += (unsigned long long)D[r];
        sum.maxdeg = max(sum.maxdeg, (unsigned)D[r]);
        if (m.planes) keep_levels<KEEP>(m.planes + (R0 + r) * planes_of<KEEP>(), nb[r], level);
      }
  }
  return nib;
}

template <int C, bool SLIMWORK, int KEEP>  // (KEEP_SHORT also where no planes are kept)
__global__ void __launch_bounds__(MULTI_ONE_THREADS, 1) k_multi_one(MultiDev m, IterLaunch il) {
  constexpr int Q = C / 4;
  const Dev& d = m.d;
  Ctl* c = d.ctl;
  if (c->done) return;
  const int level = c->k;
  const int lane = threadIdx.x & 31, lq = lane % Q;
  const int wid = blockIdx.x * (MULTI_ONE_THREADS / 32) + (threadIdx.x >> 5);
  const int nw = gridDim.x * (MULTI_ONE_THREADS / 32);
  const unsigned long long* Fp = m.F[(level - 1) & 1];
  unsigned long long* Fn = m.F[level & 1];
  const unsigned* FAp = d.fb[(level - 1) & 1];
  unsigned* FAn = d.fb[level & 1];
  if (threadIdx.x < SMEM_GUARD) ss_smem_bits[threadIdx.x] = 0u;
  // below STAGE_MIN_SLOTS slots in the previous level, reading the bits from global memory is cheaper
  const int words = level > 1 && c->prev_slots < STAGE_MIN_SLOTS ? 0 : d.smem_words;
  stage_words(FAp, words);
  stage_wait();
  const unsigned* sm = ss_smem_bits + SMEM_GUARD;
  const int sbits = words * 32;
  OneSum sum;
  for (long long b0 = wid; b0 < d.n_items; b0 += 32LL * nw) {
    const long long my_it = b0 + (long long)lane * nw;
    int4 my_item = make_int4(0, 0, 0, -1);
    long long my_start = 0;
    int a = 0;
    if (my_it < d.n_items) {
      my_item = d.items[my_it];
      a = SLIMWORK ? d.act[my_item.x] : 1;
      my_start = d.cs[my_item.x] + (long long)my_item.y * C;
    }
    unsigned todo = __ballot_sync(SS_FULL_MASK, a == 1);
    if (SLIMWORK) {  // f_k is zero on a finished chunk: clear what f_{k-2} left, twice
      unsigned carry = __ballot_sync(SS_FULL_MASK, a >= 2 && my_item.y == 0);
      while (carry) {
        const int src = __ffs(carry) - 1;
        carry &= carry - 1;
        const int chunk = __shfl_sync(SS_FULL_MASK, my_item.x, src);
        const int state = __shfl_sync(SS_FULL_MASK, a, src);
        for (int l = lane; l < C; l += 32) Fn[(long long)chunk * C + l] = 0ull;
        if (lane == 0) {
          store_bits<C>(FAn, chunk, 0u, 0u);
          d.act[chunk] = (state == 3) ? 2 : 0;
        }
      }
    }
    unsigned shortm = __ballot_sync(SS_FULL_MASK, a == 1 && my_item.w < 0 && my_item.z - my_item.y <= MULTI_SHORT);
    todo &= ~shortm;
    while (shortm) {  // short whole chunks, one group of Q lanes each
      int mysrc = -1;
#pragma unroll
      for (int g = 0; g < 32 / Q; ++g) {
        const int sidx = shortm ? __ffs(shortm) - 1 : -1;
        if (lane / Q == g) mysrc = sidx;
        shortm &= shortm - 1;
      }
      const bool own = mysrc >= 0;
      const int sl = own ? mysrc : 0;
      const int chunk = __shfl_sync(SS_FULL_MASK, my_item.x, sl);
      const int ncols = __shfl_sync(SS_FULL_MASK, my_item.z, sl) - __shfl_sync(SS_FULL_MASK, my_item.y, sl);
      const long long start = __shfl_sync(SS_FULL_MASK, my_start, sl);
      const long long R0 = (long long)chunk * C + 4 * lq;
      unsigned nib = 0;
      bool left = false;
      if (own) {
        const int4* base = reinterpret_cast<const int4*>(d.col + start) + lq;
        int4 q[MULTI_SHORT];
#pragma unroll
        for (int u = 0; u < MULTI_SHORT; ++u)
          q[u] = u < ncols ? ld_stream(base + u * Q) : make_int4(-1, -1, -1, -1);
        const ulonglong2 va = *reinterpret_cast<const ulonglong2*>(m.V + R0);
        const ulonglong2 vb = *reinterpret_cast<const ulonglong2*>(m.V + R0 + 2);
        const unsigned long long V[4] = {va.x, va.y, vb.x, vb.y};
        unsigned live = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) live |= (V[r] != ~0ull ? 1u : 0u) << r;
        unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
        one_step<MULTI_SHORT>(sm, sbits, FAp, Fp, q, live, acc);
        nib = one_post<KEEP>(m, R0, level, acc, V, Fn, sum, &left);
        sum.quads += (unsigned)ncols;
        if (lq == 0) sum.act += 1;
      }
      unsigned lo = (C <= 32 || lq < 8) ? nib << (4 * (lq & 7)) : 0u;
      unsigned hi = (C > 32 && lq >= 8) ? nib << (4 * (lq - 8)) : 0u;
      unsigned open = left;
#pragma unroll
      for (int o = 1; o < Q; o <<= 1) {
        lo |= __shfl_xor_sync(SS_FULL_MASK, lo, o);
        if (C > 32) hi |= __shfl_xor_sync(SS_FULL_MASK, hi, o);
        open |= __shfl_xor_sync(SS_FULL_MASK, open, o);
      }
      if (own && lq == 0) {
        store_bits<C>(FAn, chunk, lo, hi);
        d.act[chunk] = open ? 1 : 3;
      }
    }
    while (todo) {  // longer items, one at a time
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int chunk = __shfl_sync(SS_FULL_MASK, my_item.x, src);
      const int sidx = __shfl_sync(SS_FULL_MASK, my_item.w, src);
      const int nq = (__shfl_sync(SS_FULL_MASK, my_item.z, src) - __shfl_sync(SS_FULL_MASK, my_item.y, src)) * Q;
      const int4* base = reinterpret_cast<const int4*>(d.col + __shfl_sync(SS_FULL_MASK, my_start, src));
      const long long R0 = (long long)chunk * C + 4 * lq;
      const ulonglong2 va = *reinterpret_cast<const ulonglong2*>(m.V + R0);
      const ulonglong2 vb = *reinterpret_cast<const ulonglong2*>(m.V + R0 + 2);
      const unsigned long long V[4] = {va.x, va.y, vb.x, vb.y};
      unsigned live = 0;
#pragma unroll
      for (int r = 0; r < 4; ++r) live |= (V[r] != ~0ull ? 1u : 0u) << r;
      unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
      for (int q0 = 0; q0 < nq; q0 += 32 * MULTI_ONE_STEP) {
        int4 q[MULTI_ONE_STEP];
#pragma unroll
        for (int u = 0; u < MULTI_ONE_STEP; ++u) {
          const int at = q0 + lane + 32 * u;
          q[u] = at < nq ? ld_stream(base + at) : make_int4(-1, -1, -1, -1);
        }
        one_step<MULTI_ONE_STEP>(sm, sbits, FAp, Fp, q, live, acc);
      }
      if (lane == 0) sum.quads += (unsigned)nq;
      if (__any_sync(SS_FULL_MASK, (acc[0] | acc[1] | acc[2] | acc[3]) != 0ull)) {  // lanes that share rows
#pragma unroll
        for (int off = Q; off < 32; off <<= 1)
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[r] |= __shfl_xor_sync(SS_FULL_MASK, acc[r], off);
      }
      if (sidx >= 0) {  // SlimChunk: OR the partial rows, the last item to arrive post-processes
        unsigned long long* xa = m.xacc + (size_t)sidx * C + 4 * lane;
        if (lane < Q) {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (acc[r]) atomicOr(xa + r, acc[r]);
          __threadfence();
        }
        __syncwarp();
        int arrived = 0;
        if (lane == 0) arrived = (atomicAdd(d.arrive + sidx, 1u) == (unsigned)d.split_n[sidx] - 1u);
        if (!__shfl_sync(SS_FULL_MASK, arrived, 0)) continue;
        __threadfence();
        if (lane < Q) {
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            acc[r] = __ldcg(xa + r);
            xa[r] = 0ull;
          }
        }
        if (lane == 0) d.arrive[sidx] = 0u;
      }
      unsigned nib = 0;
      bool left = false;
      if (lane < Q) nib = one_post<KEEP>(m, R0, level, acc, V, Fn, sum, &left);
      const unsigned lo = __reduce_or_sync(SS_FULL_MASK, lane < 8 ? nib << (4 * lane) : 0u);
      const unsigned hi = C > 32 ? __reduce_or_sync(SS_FULL_MASK, (lane >= 8 && lane < 16) ? nib << (4 * (lane - 8)) : 0u) : 0u;
      const bool open = __any_sync(SS_FULL_MASK, left);
      if (lane == 0) {
        store_bits<C>(FAn, chunk, lo, hi);
        d.act[chunk] = open ? 1 : 3;
        sum.act += 1;
      }
    }
  }
  // degree sum of the rows that gained a source, each row counted once (the
  // parents pass picks its direction from it)
  unsigned long long rd = sum.rowdeg;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) rd += __shfl_down_sync(SS_FULL_MASK, rd, o);
  if (lane == 0 && rd) {
    atomicAdd(&c->new_rowdeg, rd);
    __threadfence();  // before this block counts itself done
  }
  finish_iteration_block<MULTI_ONE_THREADS>(d, sum.nw, sum.deg, 4ull * sum.quads, sum.act, sum.maxdeg, il);
}

__global__ void k_multi_init(MultiDev m, int W) {
  const Dev& d = m.d;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long words = (long long)d.n_pad * W;
  // padding rows and sources beyond k count as visited
  for (long long i = t0; i < words; i += stride) {
    const long long r = i / W;
    const int w = (int)(i % W);
    unsigned long long v = 0ull;
    if (r >= d.n) {
      v = ~0ull;
    } else {
      const int lo = 64 * w;  // sources lo .. lo+63; those >= k never exist
      if (lo >= m.k) v = ~0ull;
      else if (m.k - lo < 64) v = ~0ull << (m.k - lo);
    }
    m.V[i] = v;
    m.F[0][i] = 0ull;
    m.F[1][i] = 0ull;
  }
  for (long long i = t0; i < d.n_c; i += stride) d.act[i] = 1;
  for (long long s = t0; s < (long long)d.n_split * d.C * W; s += stride) m.xacc[s] = 0ull;
  for (long long i = t0; i < d.fb_words; i += stride) {
    d.fb[0][i] = 0u;
    d.fb[1][i] = 0u;
  }
}

__global__ void k_multi_roots(MultiDev m, int W, int* parent) {
  const Dev& d = m.d;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < m.k; s += gridDim.x * blockDim.x) {
    const int v = m.roots[s];
    const long long r = d.invperm[v];
    const unsigned long long bit = 1ull << (s & 63);
    atomicOr(m.V + r * W + s / 64, bit);
    atomicOr(m.F[0] + r * W + s / 64, bit);
    atomicOr(d.fb[0] + (r >> 5), 1u << (r & 31));
    if (m.dist && !m.planes) m.dist[(long long)v * m.k + s] = 0;
    if (parent) parent[(long long)v * m.k + s] = v;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    Ctl* c = d.ctl;
    unsigned long long rd = 0;
    for (int s = 0; s < m.k; ++s) rd += (unsigned long long)d.rdeg[d.invperm[m.roots[s]]];
    c->k = 1; c->done = 0; c->error = 0; c->variant = -1;
    c->new_count = 0; c->new_deg = 0; c->slots = 0; c->active = 0;
    c->reached = (unsigned long long)m.k; c->reached_deg = rd;
    c->total_slots = 0; c->dp_slots = 0; c->blocks_done = 0;
    c->prev_variant = -1; c->prev_slots = 0; c->prev_new = (unsigned long long)m.k; c->prev_deg = rd;
    c->prev2_new = 0; c->prev_active = 0; c->new_maxdeg = 0; c->prev_maxdeg = 0; c->units = 0; c->bunits = 0;
    c->loop_guard = 0;
    for (int v = 0; v < N_VARIANTS; ++v) c->variant_count[v] = 0;
    c->new_rowdeg = 0;
    c->prev_rowdeg = rd;  // the roots' rows (a repeated root counted again: an upper bound)
    ss_iter_stats st;
    st.frontier = m.k; st.frontier_degree = (long long)rd; st.slots = 0; st.active_chunks = 0;
    st.variant = -1; st.kernel_ns = 0;
    d.iters[0] = st;
  }
}

// Parents of the sources each row gained at `level`: (row, w) walks the row's
// neighbours in storage order (descending original id) and gives each new
// source of word w the first neighbour found in its frontier of level-1,
// stopping once every new source has one.  Each lane first walks its own row
// for up to MULTI_PAR_SHORT neighbours; rows still unresolved then are walked
// by the whole warp, 32 neighbours per step, the candidates taken in lane
// (= storage) order.  Plain stores: one lane owns each (row, word) entry.
constexpr int MULTI_PAR_SHORT = 32;
// The parents pass pushes from the previous frontier while the run grows and
// that frontier's rows carry at most nnz / MULTI_PAR_PUSH_SHARE edges.
#ifndef SS_MULTI_PAR_PUSH_SHARE
#define SS_MULTI_PAR_PUSH_SHARE 2
#endif
constexpr unsigned long long MULTI_PAR_PUSH_SHARE = SS_MULTI_PAR_PUSH_SHARE;

__global__ void __launch_bounds__(256) k_multi_parents(MultiDev m, int W, int lgW, int level, int* parent) {
  const Dev& d = m.d;
  const unsigned long long* Fp = m.F[(level - 1) & 1];
  const unsigned long long* Fn = m.F[level & 1];
  const unsigned* FAp = d.fb[(level - 1) & 1];
  const long long words = (long long)d.n_pad << lgW;
  const int lane = threadIdx.x & 31;
  const long long warp0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i0 = warp0 * 32; i0 < words; i0 += nwarps * 32) {
    const long long i = i0 + lane;
    unsigned long long rem = i < words ? Fn[i] : 0ull;
    const long long row = i >> lgW;
    const int w = (int)(i & (W - 1));
    const int v = rem ? d.perm[row] : -1;
    if (v < 0) rem = 0ull;  // padding rows never gain a source
    long long base = 0;
    int len = 0, j = 0;
    int* prow = nullptr;
    if (rem) {
      prow = parent + (long long)v * m.k + 64 * w;
      const long long chunk = row / d.C;
      base = d.cs[chunk] + (row - chunk * d.C);
      len = d.rdeg[row];  // the row's neighbours come first, padding after
      for (; j < len && j < MULTI_PAR_SHORT && rem; ++j) {
        const int u = __ldg(d.col + base + (long long)j * d.C);
        if (!((__ldg(FAp + (u >> 5)) >> (u & 31)) & 1u)) continue;
        unsigned long long f = __ldg(Fp + ((long long)u << lgW) + w) & rem;
        if (!f) continue;
        rem &= ~f;
        const int pu = __ldg(d.perm + u);
        while (f) {
          prow[__ffsll((long long)f) - 1] = pu;
          f &= f - 1;
        }
      }
    }
    unsigned pend = __ballot_sync(SS_FULL_MASK, rem != 0ull);
    while (pend) {  // long rows, one at a time, by the whole warp
      const int l = __ffs(pend) - 1;
      pend &= pend - 1;
      unsigned long long rl = __shfl_sync(SS_FULL_MASK, rem, l);
      const long long bl = __shfl_sync(SS_FULL_MASK, base, l);
      const int nl = __shfl_sync(SS_FULL_MASK, len, l);
      const int jl = __shfl_sync(SS_FULL_MASK, j, l);
      const int wl = __shfl_sync(SS_FULL_MASK, w, l);
      int* const pl = reinterpret_cast<int*>(
          __shfl_sync(SS_FULL_MASK, reinterpret_cast<unsigned long long>(prow), l));
      for (int jj = jl; jj < nl && rl; jj += 32) {
        const int jx = jj + lane;
        unsigned long long f = 0ull;
        int u = 0;
        if (jx < nl) {
          u = __ldg(d.col + bl + (long long)jx * d.C);
          if ((__ldg(FAp + (u >> 5)) >> (u & 31)) & 1u) f = __ldg(Fp + ((long long)u << lgW) + wl) & rl;
        }
        unsigned cand = __ballot_sync(SS_FULL_MASK, f != 0ull);
        const int pu = f ? __ldg(d.perm + u) : -1;
        while (cand) {  // lane order is storage order
          const int c2 = __ffs(cand) - 1;
          cand &= cand - 1;
          const unsigned long long fc = __shfl_sync(SS_FULL_MASK, f, c2) & rl;
          if (!fc) continue;
          rl &= ~fc;
          if (lane == c2) {
            unsigned long long b = fc;
            while (b) {
              pl[__ffsll((long long)b) - 1] = pu;
              b &= b - 1;
            }
          }
        }
      }
    }
  }
}

// Parents of the sources gained at `level`, pushed from the frontier of level
// - 1 (for levels whose frontier rows carry few edges).  k_multi_par_expand
// turns every row u of that frontier (summary bit set) into units of
// PUSH_UNIT neighbours; in k_multi_par_scatter one warp takes a unit and its
// lanes walk the unit's neighbours v: each source s in F[level][v] &
// F[level-1][u] has u one level closer to s than v, and atomicMax keeps the
// largest original id over all such u (parents start at -1).
__global__ void __launch_bounds__(256) k_multi_par_expand(MultiDev m, int level) {
  const Dev& d = m.d;
  const unsigned* FAp = d.fb[(level - 1) & 1];
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long words = ((long long)d.n_pad + 31) / 32;
  const long long wstride = stride & ~31LL;  // whole warps walk the summary together
  for (long long i0 = t0 - lane; i0 < words; i0 += wstride) {
    const long long i = i0 + lane;
    unsigned bits = i < words ? FAp[i] : 0u;
    while (__any_sync(SS_FULL_MASK, bits != 0u)) {
      int u = -1;
      if (bits) {
        const int b = __ffs(bits) - 1;
        bits &= bits - 1;
        u = (int)(i * 32 + b);
      }
      emit_units(d, u, lane);
    }
  }
}

__global__ void __launch_bounds__(256) k_multi_par_scatter(MultiDev m, int W, int lgW, int level,
                                                           int* parent) {
  const Dev& d = m.d;
  const unsigned long long* Fp = m.F[(level - 1) & 1];
  const unsigned long long* Fn = m.F[level & 1];
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long nunits = min((long long)d.ctl->units, d.units_cap);
  for (long long ui = wid; ui < nunits; ui += nw) {
    const int2 un = d.units[ui];
    const long long u = un.x;
    const int pu = __ldg(d.perm + u);
    const int end = min(__ldg(d.rdeg + u), un.y + PUSH_UNIT);
    const long long chunk = u / d.C;
    const long long base = __ldg(d.cs + chunk) + (u - chunk * d.C);
    for (int ww = 0; ww < W; ++ww) {
      const unsigned long long fu = __ldg(Fp + (u << lgW) + ww);
      if (!fu) continue;
      for (int j = un.y + lane; j < end; j += 32) {
        const int v = __ldg(d.col + base + (long long)j * d.C);
        unsigned long long g = __ldcg(Fn + ((long long)v << lgW) + ww) & fu;
        if (!g) continue;
        int* prow = parent + (long long)__ldg(d.perm + v) * m.k + 64 * ww;
        while (g) {
          atomicMax(prow + (__ffsll((long long)g) - 1), pu);
          g &= g - 1;
        }
      }
    }
  }
}

template <int C>
static ss_status launch_multi_one(const slimsell_graph* h, const MultiDev& m, bool slimwork,
                                  const IterLaunch& il, cudaStream_t st) {
  using Kernel = void (*)(MultiDev, IterLaunch);
  static const Kernel kernels[4] = {k_multi_one<C, false, KEEP_SHORT>, k_multi_one<C, true, KEEP_SHORT>,
                                    k_multi_one<C, false, KEEP_LONG>, k_multi_one<C, true, KEEP_LONG>};
  static std::atomic<unsigned long long> configured{0};
  if (first_on_device(configured))
    for (Kernel kern : kernels)
      SS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SS_SMEM_LIMIT_BYTES));
  const size_t smem = (size_t)(m.d.smem_words + SMEM_GUARD) * 4;
  // every SM a block, as multi_one counts on (in pull_grid, a block per 128 items of 32 warps, G(400 K, 8n)
  // gave 62 % of the SMs blocks: 529 us, 508 so)
  kernels[(slimwork ? 1 : 0) + (m.long_epoch ? 2 : 0)]<<<h->num_sms, MULTI_ONE_THREADS, smem, st>>>(m, il);
  SS_CUDA(cudaGetLastError());
  return SS_OK;
}

// Which kernel takes a one-word level.  Not k_multi_one where the last frontier was dense
// (below); where distances are written at each discovery; or where a warp of it would get
// fewer than four items, each of them a serial chain of the chunk's columns (63 sources on
// G(200001, 8n) in chunks of 64: 464 us; a thread per row 399).
static bool multi_one(const slimsell_graph* h, const MultiDev& m) {
  return !h->multi_dense && (m.planes || !m.dist) &&
         (long long)h->n_items >= 4LL * (MULTI_ONE_THREADS / 32) * h->num_sms;
}

template <int C, int W>
static ss_status launch_multi_cw(const slimsell_graph* h, const MultiDev& m, bool slimwork,
                                 const IterLaunch& il, cudaStream_t st) {
  if constexpr (C * W < 32) {
    set_error("slimsell_bfs_multi: C * ceil(k / 64) must be at least 32");
    return SS_ERR_UNSUPPORTED;
  } else {
    if constexpr (W == 1)
      if (multi_one(h, m))
        return launch_multi_one<C>(h, m, slimwork, il, st);
    using Kernel = void (*)(MultiDev, IterLaunch);
    static const Kernel kernels[6] = {k_multi_pull<C, W, false, KEEP_NOT>,   k_multi_pull<C, W, true, KEEP_NOT>,
                                      k_multi_pull<C, W, false, KEEP_SHORT>, k_multi_pull<C, W, true, KEEP_SHORT>,
                                      k_multi_pull<C, W, false, KEEP_LONG>,  k_multi_pull<C, W, true, KEEP_LONG>};
    static int grid[64][6];  // per device (zero: not measured yet)
    const int which = (slimwork ? 1 : 0) + (m.planes ? (m.long_epoch ? 4 : 2) : 0);
    int& g = grid[h->device & 63][which];
    if (!g) {
      int b = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernels[which], C * W, 0);
      if (SS_MULTI_BLOCKS_PER_SM > 0) b = std::min(b, SS_MULTI_BLOCKS_PER_SM);
      g = (b > 0 ? b : 1) * h->num_sms;
    }
    kernels[which]<<<g, C * W, 0, st>>>(m, il);
    SS_CUDA(cudaGetLastError());
    return SS_OK;
  }
}

template <int C>
static ss_status launch_multi_c(const slimsell_graph* h, const MultiDev& m, int W, bool slimwork,
                                const IterLaunch& il, cudaStream_t st) {
  switch (W) {
    case 1: return launch_multi_cw<C, 1>(h, m, slimwork, il, st);
    case 2: return launch_multi_cw<C, 2>(h, m, slimwork, il, st);
    case 4: return launch_multi_cw<C, 4>(h, m, slimwork, il, st);
    case 8: return launch_multi_cw<C, 8>(h, m, slimwork, il, st);
    default: return launch_multi_cw<C, 16>(h, m, slimwork, il, st);
  }
}

static ss_status launch_multi(const slimsell_graph* h, const MultiDev& m, int W, bool slimwork,
                              const IterLaunch& il, cudaStream_t st) {
  switch (h->C) {
    case 8: return launch_multi_c<8>(h, m, W, slimwork, il, st);
    case 16: return launch_multi_c<16>(h, m, W, slimwork, il, st);
    case 32: return launch_multi_c<32>(h, m, W, slimwork, il, st);
    default: return launch_multi_c<64>(h, m, W, slimwork, il, st);
  }
}

// Which kernel takes the next one-word level (from the counters just read): where the
// frontier's rows hold over 1 / MULTI_DENSE_SHARE of the edges, most lookups hit, and what
// counts is how many of the gathered words L1 holds; the block kernel leaves it all of L1,
// k_multi_one uses it for the bits (64 sources on Kronecker 22, the dense level: 615 us,
// 1155 in k_multi_one).
constexpr unsigned long long MULTI_DENSE_SHARE = 8;
static bool multi_dense(const slimsell_graph* h) {
  return h->h_ctl->prev_rowdeg * MULTI_DENSE_SHARE > (unsigned long long)h->nnz;
}

// Multi-source scratch, grown on demand and kept with the handle.
static ss_status ensure_multi_scratch(slimsell_graph* h, int W) {
  if (h->multi_w >= W) return SS_OK;
  drop_planes(h);
  void* ptrs[] = {h->mF[0], h->mF[1], h->mV, h->mxacc, h->mroots};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  h->mF[0] = h->mF[1] = h->mV = h->mxacc = nullptr;
  h->mroots = nullptr;
  h->multi_w = 0;
  const size_t words = (size_t)h->n_pad * W;
  ss_status s;
  for (int b = 0; b < 2; ++b)
    if ((s = dmalloc(h, (void**)&h->mF[b], sizeof(unsigned long long) * words)) != SS_OK) return s;
  if ((s = dmalloc(h, (void**)&h->mV, sizeof(unsigned long long) * words)) != SS_OK) return s;
  const size_t ns = (size_t)(h->n_split > 0 ? h->n_split : 1) * h->C * W;
  if ((s = dmalloc(h, (void**)&h->mxacc, sizeof(unsigned long long) * ns)) != SS_OK) return s;
  if ((s = dmalloc(h, (void**)&h->mroots, sizeof(int) * 1024)) != SS_OK) return s;
  h->multi_w = W;
  return SS_OK;
}

static size_t plane_bytes(const slimsell_graph* h, bool long_epoch) {
  return sizeof(unsigned long long) * (long_epoch ? MULTI_LONG_PLANES : MULTI_SHORT_PLANES) * (size_t)h->n_pad *
         (size_t)h->multi_w;
}

// The planes stay with the handle from call to call, but no other allocation of it fails for
// them (dmalloc).
bool drop_planes(slimsell_graph* h) {
  bool any = false;
  for (int i = 0; i < 2; ++i)
    if (h->mplanes[i]) {
      cudaFree(h->mplanes[i]);
      h->mplanes[i] = nullptr;
      h->device_bytes -= (long long)plane_bytes(h, i == 1);
      any = true;
    }
  return any;
}

// Planes of the next epoch, cleared; allocated by the first call that wants them.
// SS_ERR_OOM: the caller does with shorter epochs, or without.
static ss_status next_planes(slimsell_graph* h, MultiDev* m, bool long_epoch, cudaStream_t st) {
  unsigned long long*& p = h->mplanes[long_epoch ? 1 : 0];
  if (!p) {
    const ss_status s = dmalloc(nullptr, (void**)&p, plane_bytes(h, long_epoch));
    if (s != SS_OK) {
      set_error("");  // (the call goes on)
      return s;
    }
    h->device_bytes += (long long)plane_bytes(h, long_epoch);
  }
  m->planes = p;
  m->long_epoch = long_epoch ? 1 : 0;
  SS_CUDA(cudaMemsetAsync(p, 0, sizeof(unsigned long long) * (long_epoch ? MULTI_LONG_PLANES : MULTI_SHORT_PLANES) *
                                    (size_t)m->plane_words, st));
  return SS_OK;
}

// Whether the epoch under way ends with `level`, and the last level before it.
static bool epoch_ends(const MultiDev& m, int level) {
  return m.long_epoch ? (level - MULTI_EPOCH) % MULTI_EPOCH_LONG == 0 : level % MULTI_EPOCH == 0;
}
static int epoch_base(const MultiDev& m, int level) {
  return m.long_epoch ? MULTI_EPOCH + (level - 1 - MULTI_EPOCH) / MULTI_EPOCH_LONG * MULTI_EPOCH_LONG
                      : (level - 1) / MULTI_EPOCH * MULTI_EPOCH;
}

// Write the distances of the epoch that ends with `level`, and clear planes for the next one
// when more levels follow.
static ss_status write_levels(slimsell_graph* h, MultiDev* m, int W, int level, bool more, cudaStream_t st) {
  int lgW = 0;
  while ((1 << lgW) < W) ++lgW;
  const int base = epoch_base(*m, level);
  if (m->long_epoch) k_multi_levels<MULTI_LONG_PLANES><<<16 * h->num_sms, 256, 0, st>>>(*m, W, lgW, base);
  else k_multi_levels<MULTI_SHORT_PLANES><<<16 * h->num_sms, 256, 0, st>>>(*m, W, lgW, base);
  if (base == 0) k_multi_root_levels<<<(m->k + 255) / 256, 256, 0, st>>>(*m);
  SS_CUDA(cudaGetLastError());
  if (!more) return SS_OK;
  // (long epochs begin after the first short one or not at all)
  const ss_status s = next_planes(h, m, m->long_epoch || level == MULTI_EPOCH, st);
  return s == SS_ERR_OOM ? next_planes(h, m, false, st) : s;
}

// Level-by-level multi-source BFS for the passes built on it (betweenness
// centrality): seeds k sources (device ids, checked by the caller) and returns
// the view of the handle's multi-source state; multi_level then runs one level
// (SlimWork pull) and reports whether it discovered nothing.  The frontier words
// of level L are m->F[L & 1] (W words per row) until level L + 2 overwrites them.
// Optional events are recorded around the level's kernel.
ss_status multi_start(slimsell_graph* h, const int32_t* d_roots, int k, cudaStream_t st, MultiDev* m,
                      int* W_out) {
  int W = 1;
  while (64 * W < k) W *= 2;
  while (h->C * W < 32) W *= 2;
  if (h->pending) SS_CUDA(cudaEventSynchronize(h->ev_done));
  h->pending = 0;
  h->multi_dense = false;
  ss_status s = ensure_multi_scratch(h, W);
  if (s != SS_OK) return s;
  SS_CUDA(cudaMemcpyAsync(h->mroots, d_roots, sizeof(int) * (size_t)k, cudaMemcpyDeviceToDevice, st));
  m->d = h->dev();
  m->d.reach_cap = (unsigned long long)h->n * (unsigned long long)k;
  m->F[0] = h->mF[0];
  m->F[1] = h->mF[1];
  m->V = h->mV;
  m->xacc = h->mxacc;
  m->dist = nullptr;
  m->vec_dist = 0;
  m->planes = nullptr;
  m->plane_words = 0;
  m->long_epoch = 0;
  m->roots = h->mroots;
  m->k = k;
  k_multi_init<<<8 * h->num_sms, 256, 0, st>>>(*m, W);
  k_multi_roots<<<(k + 255) / 256, 256, 0, st>>>(*m, W, nullptr);
  SS_CUDA(cudaGetLastError());
  *W_out = W;
  return SS_OK;
}

ss_status multi_level(slimsell_graph* h, const MultiDev& m, int W, cudaStream_t st, bool* done,
                      cudaEvent_t before, cudaEvent_t after) {
  if (before) SS_CUDA(cudaEventRecord(before, st));
  ss_status s = launch_multi(h, m, W, true, IterLaunch{SS_V_SLIMWORK, 0, 0}, st);
  if (s != SS_OK) return s;
  if (after) SS_CUDA(cudaEventRecord(after, st));
  SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  if (h->h_ctl->error) {
    set_error("multi-source BFS: device error flags %d", h->h_ctl->error);
    return SS_ERR_CUDA;
  }
  *done = h->h_ctl->done != 0;
  h->multi_dense = multi_dense(h);
  return SS_OK;
}

}  // namespace ss

extern "C" ss_status slimsell_bfs_multi(slimsell_handle h, const int32_t* d_roots, int32_t k,
                                        int32_t policy, int32_t* d_dist, void* stream) {
  return slimsell_bfs_multi_parents(h, d_roots, k, policy, d_dist, nullptr, stream);
}

extern "C" ss_status slimsell_bfs_multi_parents(slimsell_handle h, const int32_t* d_roots, int32_t k,
                                                int32_t policy, int32_t* d_dist, int32_t* d_parent,
                                                void* stream) {
  using namespace ss;
  set_error("");
  if (!h || !d_roots) {
    set_error("slimsell_bfs_multi: NULL argument");
    return SS_ERR_INVALID;
  }
  h->values_semiring = -1;
  if (k < 1 || k > 1024) {
    set_error("slimsell_bfs_multi: k must be in [1, 1024] (got %d)", k);
    return SS_ERR_INVALID;
  }
  if (policy != SS_V_FULL && policy != SS_V_SLIMWORK) {
    set_error("slimsell_bfs_multi: policy must be SS_V_FULL or SS_V_SLIMWORK");
    return SS_ERR_INVALID;
  }
  int W = 1;
  while (64 * W < k) W *= 2;
  while (h->C * W < 32) W *= 2;  // a block needs a full warp; extra words hold no source
  cudaStream_t st = (cudaStream_t)stream;
  std::vector<int> roots((size_t)k);
  SS_CUDA(cudaMemcpyAsync(roots.data(), d_roots, sizeof(int) * (size_t)k, cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  for (int s = 0; s < k; ++s)
    if (roots[(size_t)s] < 0 || roots[(size_t)s] >= h->n) {
      set_error("slimsell_bfs_multi: root %d of source %d out of range", roots[(size_t)s], s);
      return SS_ERR_INVALID;
    }
  if (h->pending) SS_CUDA(cudaEventSynchronize(h->ev_done));
  h->pending = 0;
  ss_status s = ensure_multi_scratch(h, W);
  if (s != SS_OK) return s;
  SS_CUDA(cudaMemcpyAsync(h->mroots, d_roots, sizeof(int) * (size_t)k, cudaMemcpyDeviceToDevice, st));
  MultiDev m;
  m.d = h->dev();
  m.d.reach_cap = (unsigned long long)h->n * (unsigned long long)k;
  m.F[0] = h->mF[0];
  m.F[1] = h->mF[1];
  m.V = h->mV;
  m.xacc = h->mxacc;
  m.dist = d_dist;
  m.planes = nullptr;
  m.plane_words = (long long)h->n_pad * W;
  m.long_epoch = 0;
  if (d_dist && multi_planes(h, k, W)) {
    s = next_planes(h, &m, false, st);
    if (s != SS_OK && s != SS_ERR_OOM) return s;
  }
  m.vec_dist = (k % 4 == 0) && ((reinterpret_cast<uintptr_t>(d_dist) & 15u) == 0);
  m.roots = h->mroots;
  m.k = k;
  const bool prof = h->profiling != 0;
  h->iter_ns.clear();
  double iter_ms = 0.0;
  if (prof) SS_CUDA(cudaEventRecord(h->ev_c, st));
  if (d_dist && !m.planes) SS_CUDA(cudaMemsetAsync(d_dist, 0xff, sizeof(int) * (size_t)h->n * (size_t)k, st));
  if (d_parent) SS_CUDA(cudaMemsetAsync(d_parent, 0xff, sizeof(int) * (size_t)h->n * (size_t)k, st));
  k_multi_init<<<8 * h->num_sms, 256, 0, st>>>(m, W);
  k_multi_roots<<<(k + 255) / 256, 256, 0, st>>>(m, W, d_parent);
  int lgW = 0;
  while ((1 << lgW) < W) ++lgW;
  SS_CUDA(cudaGetLastError());
  if (d_parent) {  // the first frontier's edges (the roots' rows), for the parents pass
    SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
    SS_CUDA(cudaStreamSynchronize(st));
  }
  const IterLaunch il{policy, 0, 0};
  h->multi_dense = false;
  const long long max_iter = (long long)h->n + 2;
  for (long long it = 0;; ++it) {
    if (it > max_iter) {
      set_error("slimsell_bfs_multi: no convergence after %lld iterations", it);
      return SS_ERR_CUDA;
    }
    if (prof) SS_CUDA(cudaEventRecord(h->ev_a, st));
    s = launch_multi(h, m, W, policy == SS_V_SLIMWORK, il, st);
    if (s != SS_OK) return s;
    if (d_parent) {  // parents of the sources gained at this level
      // push from the previous frontier while the run grows and that frontier's
      // rows carry at most 1 / MULTI_PAR_PUSH_SHARE of the edges (the gaining
      // rows would have to search deep into their rows for it); once the
      // frontiers are dense or shrinking, the gaining rows find their parents
      // within a few neighbours and walk (measured on Kronecker 22, k = 64 ..
      // 1024: the push wins levels 1 and 2 by 7-70x, the walk every later level)
      const Ctl& hc = *h->h_ctl;  // counters read after the previous level
      const bool growing = hc.prev_new >= hc.prev2_new;
      if (growing && hc.prev_rowdeg * MULTI_PAR_PUSH_SHARE <= (unsigned long long)h->nnz) {
        SS_CUDA(cudaMemsetAsync(&h->ctl->units, 0, sizeof(unsigned long long), st));
        k_multi_par_expand<<<8 * h->num_sms, 256, 0, st>>>(m, (int)(it + 1));
        k_multi_par_scatter<<<8 * h->num_sms, 256, 0, st>>>(m, W, lgW, (int)(it + 1), d_parent);
      } else
        k_multi_parents<<<8 * h->num_sms, 256, 0, st>>>(m, W, lgW, (int)(it + 1), d_parent);
      SS_CUDA(cudaGetLastError());
    }
    if (prof) SS_CUDA(cudaEventRecord(h->ev_b, st));
    SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
    SS_CUDA(cudaStreamSynchronize(st));
    if (prof) {
      float ms = 0.f;
      SS_CUDA(cudaEventElapsedTime(&ms, h->ev_a, h->ev_b));
      iter_ms += ms;
      h->iter_ns.push_back((int)(ms * 1.0e6f));
    }
    const bool done = h->h_ctl->done != 0;
    h->multi_dense = multi_dense(h);
    if (m.planes && (done || epoch_ends(m, (int)(it + 1)))) {
      if (prof) SS_CUDA(cudaEventRecord(h->ev_a, st));
      if ((s = write_levels(h, &m, W, (int)(it + 1), !done, st)) != SS_OK) return s;
      if (prof) {  // the epoch's distance writes are work of its last level
        SS_CUDA(cudaEventRecord(h->ev_b, st));
        SS_CUDA(cudaEventSynchronize(h->ev_b));
        float ms = 0.f;
        SS_CUDA(cudaEventElapsedTime(&ms, h->ev_a, h->ev_b));
        iter_ms += ms;
        h->iter_ns.back() += (int)(ms * 1.0e6f);
      }
    }
    if (done) break;
  }
  if (prof) SS_CUDA(cudaEventRecord(h->ev_d, st));
  SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaEventRecord(h->ev_done, st));
  h->last.semiring = SS_BOOLEAN;
  h->last.iter_kernel_ms = iter_ms;
  h->last.total_ms = 0.0;
  h->pending = 1;
  ss_run_stats tmp;
  return slimsell_get_run_stats(h, &tmp, nullptr, 0);
}
