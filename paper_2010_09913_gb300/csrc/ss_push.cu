// Compacted-frontier push iteration on the SlimSell layout (the direction-
// optimising work avoidance that Section V calls orthogonal to SlimSell and
// implementable on top of it).  It computes exactly what the pull iteration
// computes -- new rows, their largest-id frontier neighbour, the real-semiring
// sum of frontier values -- by scattering from the frontier instead of
// gathering into every row:
//
//   k_push_expand   clears the touched map and turns each level-(k-1) vertex
//                   (read from the frontier bitmap) into work units of
//                   PUSH_UNIT neighbours;
//   k_push_scatter  one warp per unit reads the vertex's row (column-major, so
//                   with stride C) and, for every unvisited neighbour, folds in
//                   the parent by an atomicMax on its claim word's lower half, the real
//                   value by atomicAdd and a touched bit by atomicOr (reductions:
//                   no result is read);
//   k_push_post     walks the touched words: a touched word becomes the
//                   frontier word of level k (fb[k&1] held level k-2, which is
//                   overwritten) and joins the visited bits, and each touched row
//                   gets its level and value; the scratch is reset and the iteration
//                   tail runs.
#include <algorithm>
#include <climits>

#include <cooperative_groups.h>

#include "ss_device.cuh"

namespace ss {

namespace cg = cooperative_groups;

constexpr int PUSH_THREADS = 256;

// Emit the block units (chunk, first column) of chunk i, warp-aggregated; all
// lanes call, lanes with i < 0 emit nothing.
template <int C>
__device__ __forceinline__ void emit_block_units(const Dev& d, long long i, int lane) {
  constexpr int COLS = PUSH_BLOCK_SLOTS / C;
  const int cl = (i >= 0) ? d.cl[i] : 0;
  const unsigned nu = (unsigned)((cl + COLS - 1) / COLS);
  unsigned incl = nu;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(SS_FULL_MASK, incl, o);
    if (lane >= o) incl += t;
  }
  const unsigned total = __shfl_sync(SS_FULL_MASK, incl, 31);
  unsigned long long base = 0;
  if (lane == 31 && total) base = atomicAdd(&d.ctl->bunits, (unsigned long long)total);
  base = __shfl_sync(SS_FULL_MASK, base, 31);
  const unsigned long long first = base + incl - nu;
  if (first + nu > (unsigned long long)d.bunits_cap) {  // cannot happen: the capacity covers every chunk
    if (nu) atomicOr(&d.ctl->error, 2);
    return;
  }
  for (unsigned q = 0; q < nu; ++q) d.bunits[first + q] = make_int2((int)i, (int)(q * COLS));
}

// The frontier f_{k-1} as work: walked one chunk (one block of C rows, the
// layout's own block size) per lane.  With push_blocks on, a chunk whose block
// holds at least C/4 frontier rows (all non-empty blocks with push_blocks = 2)
// becomes block units that read whole columns of the chunk with coalesced
// loads, the block-sparse frontier; the rows of sparser blocks become vertex
// units that read one row each (stride C).  Also clears the touched map.
template <int C>
__global__ void __launch_bounds__(PUSH_THREADS) k_push_expand(Dev d) {
  const Ctl* c = d.ctl;
  if (c->done) return;
  const int k = c->k;
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long words = ((long long)d.n_pad + 31) / 32;
  for (long long w = t0; w < words; w += stride) d.touched[w] = 0u;
  const long long wstride = stride & ~31LL;  // whole warps walk the chunks together
  const unsigned* fbm = d.fb[(k - 1) & 1];
  for (long long i0 = t0 - lane; i0 < d.n_c; i0 += wstride) {
    const long long i = i0 + lane;
    unsigned long long bits = i < d.n_c ? chunk_bits<C>(fbm, i) : 0ull;
    const int pc = __popcll(bits);
    const bool block = bits && (d.push_blocks == 2 || (d.push_blocks == 1 && pc >= C / 4));
    if (__any_sync(SS_FULL_MASK, block)) emit_block_units<C>(d, block ? i : -1, lane);
    if (block) bits = 0ull;
    while (__any_sync(SS_FULL_MASK, bits != 0ull)) {
      int u = -1;
      if (bits) {
        const int b = __ffsll((long long)bits) - 1;
        bits &= bits - 1;
        u = (int)(i * C + b);
      }
      emit_units(d, u, lane);
    }
  }
}

// Fold the frontier row with original id `id` (real value val) into neighbour v unless v
// was visited at an earlier level.  Most neighbours of a large level are, hubs above all,
// so that is asked of the visited bitmap, which stays as it is until the level's post and
// is small enough for L1.  Among the rows of this level the largest id wins, so the claim
// word's lower half (0 before the level) takes a 32-bit max and k_push_post adds the level;
// whoever finds the half empty marks the row as touched (the first to write it did).
// Bound by the scattered accesses to L2, three an edge when every edge asked a 64-bit
// claim word, changed it by a 64-bit max and asked the touched map: Kronecker 22, the
// level of 116 M edges, 1,149 us, and 351 so; G(2.8 M, 8n), 13.6 M edges, 331 and 210.
// (With 32-bit levels and parents of their own, 553 and 307.)
template <int SR>
__device__ __forceinline__ void push_fold(const Dev& d, int v, int id, float val) {
  const unsigned bit = 1u << (v & 31);
  if (__ldg(d.vis + (v >> 5)) & bit) return;
  unsigned* best = reinterpret_cast<unsigned*>(parent_half(d, v));
  // it only grows, so a stale read can only cause a redundant atomic, never a missed one
  const unsigned seen = *(volatile const unsigned*)best, mine = (unsigned)(id + 1);
  if (seen < mine) atomicMax(best, mine);
  if (SR == SS_REAL) atomicAdd(d.psum + v, val);
  if (seen == 0u) atomicOr(d.touched + (v >> 5), bit);
}

template <int SR, int C>
__global__ void __launch_bounds__(PUSH_THREADS) k_push_scatter(Dev d) {
  const Ctl* c = d.ctl;
  if (c->done) return;
  const long long nunits = min((long long)c->units, d.units_cap);
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  unsigned long long my_slots = 0;
  for (long long ui = wid; ui < nunits; ui += nw) {
    const int2 un = d.units[ui];
    const int u = un.x;
    const int deg = d.rdeg[u];
    const int chunk = u / C, l = u % C;
    const int* rowp = d.col + d.cs[chunk] + l;
    const int id = __ldg(d.perm + u);
    const float val = (SR == SS_REAL) ? d.fr[u] : 0.0f;
    const int jend = min(un.y + PUSH_UNIT, deg);
    for (int j = un.y + lane; j < jend; j += 32) {
      const int v = __ldg(rowp + (long long)j * C);
      ++my_slots;
      push_fold<SR>(d, v, id, val);
    }
  }
  // block units: columns [j0, j0 + COLS) of a chunk whose frontier block is
  // dense, read as 16-byte quads (lane l meets rows 4 (l mod C/4) .. + 3 in
  // every column); only the block's frontier rows fold their neighbours in
  {
    constexpr int Q = C / 4;
    constexpr int COLS = PUSH_BLOCK_SLOTS / C;
    const long long nb = min((long long)c->bunits, d.bunits_cap);
    const unsigned* fbm = d.fb[(c->k - 1) & 1];
    const int lq = lane % Q;
    for (long long bi = wid; bi < nb; bi += nw) {
      const int2 un = d.bunits[bi];
      const long long chunk = un.x;
      const unsigned mb = (unsigned)(chunk_bits<C>(fbm, chunk) >> (4 * lq)) & 0xFu;
      const int ncols = min(COLS, d.cl[chunk] - un.y);
      if (lane == 0) my_slots += (unsigned long long)ncols * C;
      if (!mb) continue;  // none of this lane's rows is in the frontier
      const long long r0 = chunk * C + 4 * lq;
      int origs[4];
      float vals[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        origs[r] = (mb >> r & 1u) ? __ldg(d.perm + r0 + r) : -1;
        vals[r] = (SR == SS_REAL && (mb >> r & 1u)) ? d.fr[r0 + r] : 0.0f;
      }
      const int4* base = reinterpret_cast<const int4*>(d.col + d.cs[chunk] + (long long)un.y * C) + lq;
      for (int j = lane / Q; j < ncols; j += 32 / Q) {
        const int4 q = __ldcs(base + (long long)j * Q);
        const int cc[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if ((mb >> r & 1u) && cc[r] >= 0) push_fold<SR>(d, cc[r], origs[r], vals[r]);
      }
    }
  }
  __shared__ unsigned long long red[PUSH_THREADS / 32];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) my_slots += __shfl_down_sync(SS_FULL_MASK, my_slots, off);
  if (lane == 0) red[threadIdx.x >> 5] = my_slots;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long s = 0;
    for (int w = 0; w < PUSH_THREADS / 32; ++w) s += red[w];
    if (s) atomicAdd(&d.ctl->slots, s);
  }
}

template <int SR>
__global__ void __launch_bounds__(PUSH_THREADS) k_push_post(Dev d, IterLaunch il) {
  const Ctl* c = d.ctl;
  if (c->done) return;
  const int k = c->k;
  unsigned* fbk = d.fb[k & 1];
  const long long words = ((long long)d.n_pad + 31) / 32;
  unsigned long long nw = 0, deg = 0;
  unsigned maxdeg = 0;
  for (long long w = (long long)blockIdx.x * blockDim.x + threadIdx.x; w < words;
       w += (long long)gridDim.x * blockDim.x) {
    unsigned bits = d.touched[w];
    fbk[w] = bits;  // f_k: exactly the rows first reached now
    if (bits) d.vis[w] |= bits;
    while (bits) {
      const int b = __ffs(bits) - 1;
      bits &= bits - 1;
      const int v = (int)(w * 32 + b);
      reinterpret_cast<unsigned*>(d.claim + v)[1] = claim_upper(k);
      if (SR == SS_REAL) {
        d.fr[v] = d.psum[v];
        d.psum[v] = 0.0f;
      }
      const int dv = d.rdeg[v];
      ++nw;
      deg += (unsigned long long)dv;
      maxdeg = max(maxdeg, (unsigned)dv);
    }
  }
  finish_iteration_block<PUSH_THREADS>(d, nw, deg, 0ull, 0ull, maxdeg, il);
}

// ---------------------------------------------------------------------------
// Cluster push for small frontiers: one thread-block cluster (16 CTAs of 512
// threads where the device can place it, else 8) runs level after level inside
// one launch, with no kernel boundary and no bitmap walk per level.
//
// The frontier lives in shared memory as entries of at most LOCAL_EDGES edges
// (start in col, edge count, original id, row); rows of more than LOCAL_LONG edges
// become entries of LOCAL_UNIT edges that a warp walks together.  A thread takes an
// entry, loads its neighbours, claims each with one atomicMax on its claim word
// (old value 0: this thread discovered it; words of earlier levels are larger and
// never change; the word ends with this level and the largest id among the
// frontier neighbours, the parent), and writes each discovered row's entries
// straight into the shared memory of the CTA that takes them in the next level
// (distributed shared memory).  Where an entry goes follows from its number among
// the entries its CTA has made (round-robin over the CTAs, one segment per making
// CTA), so no count is needed before the placing and a level has one cluster
// barrier: the claim word needs no second step after the claims are final.
//
// A level is a chain of latencies (columns, claims, row data, barrier), and the
// barrier with its release of the level's global writes is the longest.  While levels
// have up to SOLO_UP edges they are therefore run by rank 0 alone, entries in its own shared
// memory, block barriers only, while the others wait at a cluster barrier until it
// spreads the entries again or ends the launch.  Lattice 4096^2 (6,154 levels): 4.5 us a
// level, 7.2 with two cluster barriers a level; 96^2, mostly rank 0 alone, about 2.4 us.
//
// A level of more edges than the cluster has threads is bound not by that chain but by its
// scattered accesses, on graphs past L2 to DRAM.  Such a level (`late`) therefore reads row data
// of new rows only, after the claims, and asks for no columns ahead of the next level.  Lattice
// 8192^2 (14,900 levels), us a level of 8 .. 16 K edges / 16 .. 24 K / 24 .. 32 K, and a run:
// 7.1 / 13.3 / 19.8, 167 ms, with every neighbour's row data up to 32 K edges;
// 5.8 / 10.0 / 15.2, 134 ms, with new rows' alone; 5.8 / 9.4 / 13.4, 124 ms, so (7.8 / 10.3 / 12.2,
// 139 ms, by the two-barrier form).  4096^2: 31.0 ms, 28.2 so; from 4 K edges on 28.1.
//
// Every active CTA takes the same exits (counters reach every CTA through
// distributed shared memory); rank 0 keeps the control block in shared memory and
// writes it back.  Frontier bits are kept in no level: a launch clears those of its
// first frontier, and when it hands back it sets those of the last, as the
// grid-wide variants expect them (fb[(k-1)&1] = level k-1, fb[k&1] = 0).
// ---------------------------------------------------------------------------
#ifndef SS_LOCAL_THREADS
#define SS_LOCAL_THREADS 512
#endif
constexpr int LOCAL_THREADS = SS_LOCAL_THREADS;
constexpr int LOCAL_EDGES = 4;      // edges a thread takes at once, and of one entry of a short row
constexpr int LOCAL_LONG = 64;      // longer rows are cut into units of
constexpr int LOCAL_UNIT = 128;     // edges, walked by a warp
constexpr int LOCAL_ENTRIES = 6144; // entries a CTA holds of one level
constexpr int SOLO_UP = SS_LOCAL_SOLO_UP;      // rank 0 goes on alone after a level of up to this many edges
constexpr int SOLO_DOWN = SS_LOCAL_SOLO_DOWN;  // the cluster leaves the next level to it after one of this many
constexpr int CTL_WORDS = (int)(sizeof(Ctl) / sizeof(unsigned));
static_assert(sizeof(Ctl) % sizeof(unsigned) == 0, "control block copied as words");
static_assert(SOLO_DOWN <= SOLO_UP && SOLO_UP <= LOCAL_ENTRIES, "the first solo level fits one CTA");

struct LocalPub {             // what a CTA tells the others about a level
  int nent;                   // entries it has made
  int nnew;                   // vertices it has discovered
  unsigned md;                // their largest degree
  int drop;                   // a vertex found no room (the level goes back to the grid)
  unsigned nd_lo, nd_hi;      // their degree sum, nd_lo + nd_hi * 2^20 (32-bit shared atomics are native)
};

struct __align__(16) LocalEntry {
  unsigned long long edges;   // start of the entry's first edge in col, edge count << 44
  int orig;                   // original id of its row (parent candidate)
  int row;                    // its row; -1 - row for all but the row's first entry
};

struct LocalMsg {             // rank 0 to the waiting CTAs, at the end of its solo levels
  int k, exit, handback, dropped;
  unsigned long long nf, E, reached, reached_deg;
};

struct LocalSmem {
  Ctl ctl;                                // rank 0: the control block
  LocalEntry ent[2][LOCAL_ENTRIES];       // by level parity
  LocalPub mine[3];                       // this CTA's counters, by level modulo 3
  LocalPub all[2][SS_LOCAL_CLUSTER_MAX];  // every CTA's
  unsigned placed[2];                     // edges of the long rows this CTA has placed
  LocalMsg msg;
};
static_assert(sizeof(LocalSmem) <= 227 * 1024, "cluster push shared memory");
static_assert(LOCAL_THREADS / 32 >= SS_LOCAL_CLUSTER_MAX, "a warp for every segment of a slice");

extern __shared__ __align__(16) unsigned char ss_local_smem[];

// How the entries of a level lie: made by rank 0 alone or by every CTA, for rank 0
// alone or for every CTA.  A making CTA owns one segment of every taking CTA.
struct LocalLay {
  bool from_one, to_one;
  __device__ __forceinline__ int cap(int lg) const { return from_one ? LOCAL_ENTRIES : LOCAL_ENTRIES >> lg; }
  // entries that CTA `rank` takes of the nent ones CTA r has made
  __device__ __forceinline__ int count(int r, int nent, int rank, int lg) const {
    if (from_one && r != 0) return 0;
    if (to_one) return rank == 0 ? min(nent, cap(lg)) : 0;
    const int G = 1 << lg, e0 = (rank - r) & (G - 1);
    return nent > e0 ? min((nent - e0 + G - 1) >> lg, cap(lg)) : 0;
  }
};

// Call f(index, valid) for this CTA's entries of parity p: the threads of a warp together;
// invalid past the last entry.
// (made: how many rank 0 has made, where it alone did).
template <class F>
__device__ __forceinline__ void local_entries(const LocalSmem& S, const LocalLay& lay, int made, int p, int rank,
                                              int lg, F f) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NW = LOCAL_THREADS / 32;
  const int nseg = lay.from_one ? 1 : 1 << lg;
  const int nent = lane < nseg ? lay.count(lane, lay.from_one ? made : S.all[p][lane].nent, rank, lg) : 0;
  const int total = (int)__reduce_add_sync(SS_FULL_MASK, (unsigned)nent);
  const int most = (int)__reduce_max_sync(SS_FULL_MASK, (unsigned)nent);
  // Each segment has warps of its own, and entry after entry goes to another of them, so that a
  // few long ones do not queue in one.  Uneven segments are one list for all the warps instead:
  // in a level made by a few CTAs alone (three units of a hub) as few warps had all the work
  // (282 rows of 92,934 edges on Kronecker 14: 81 us, 22 so), and so are segments of more
  // entries than their warps' lanes, a few of which would be a second round (levels of 24 .. 32 K
  // edges on lattice 8192^2: 14.0 us, 13.4 so).  The search for an entry's segment made a
  // lattice's small levels 8 % longer where it was always done.
  const bool list = most >= 8 && (most * nseg > 2 * total || most > 32 * (NW / nseg));
  int incl = nent;
  if (list) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(SS_FULL_MASK, incl, o);
      if (lane >= o) incl += t;
    }
  }
  const int before = incl - nent;
  const int wps = list ? NW : NW / nseg;  // warps of a segment
  const int own = warp / wps;
  const int n = list ? total : __shfl_sync(SS_FULL_MASK, nent, own);
  for (int i0 = warp % wps; i0 < n; i0 += wps * 32) {
    const int i = i0 + lane * wps;
    int seg = own, at = i;
    if (list) {
      seg = 0;  // segments that end at or before entry i
      for (int step = nseg >> 1; step; step >>= 1)
        if (__shfl_sync(SS_FULL_MASK, incl, seg + step - 1) <= i) seg += step;
      at -= __shfl_sync(SS_FULL_MASK, before, seg);
    }
    f(seg * lay.cap(lg) + at, i < n);
  }
}

// Selector features of the iterations after levels k0 .. k1 run in this launch
// (the decide kernel did not run before them), from the per-level totals the
// launch recorded; rank 0's threads, one level each, when the launch ends.
__device__ __forceinline__ void local_features(const Dev& d, int k0, int k1) {
  __syncthreads();  // the last level's totals are in place
  for (int k = k0 + (int)threadIdx.x; k <= k1 && k + 1 < d.iter_cap; k += LOCAL_THREADS) {
    const unsigned long long* ls = d.lstat + (size_t)k * SS_LSTAT;
    float f[SS_SELECTOR_FEATURES];
    features_of(d, k + 1, ls[0], ls[1], ls[4], ls[5], (unsigned)ls[2], ls[6], f);
    store_features(d, k + 1, f);
  }
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// A level's placing: where the rows that this CTA discovers go.
template <int C>
struct LocalPlace {
  const Dev& d;
  LocalSmem& S;
  cg::cluster_group& cl;
  LocalPub* mine;
  int k, p, rank, lg;
  LocalLay lay;
  bool late;   // a level of more edges than the cluster has threads
  bool first;  // the launch's own entries: numbered through one counter for all CTAs, as if rank 0 made them
  // a row without room: the level is handed back, as a bitmap, where its bit is set at once
  __device__ __forceinline__ void drop(int x) {
    mine->drop = 1;
    atomicOr(d.fb[p] + (x >> 5), 1u << (x & 31));
    atomicOr(d.vis + (x >> 5), 1u << (x & 31));
  }
  // Unit u of a row as entry number e; false (and the row dropped) without room: what fits of
  // the row is placed all the same, it is then set twice.
  __device__ __forceinline__ bool put(int x, long long bx, int deg, int og, int per, int u, int e, int seg, int cap,
                                      int from) {
    const int slot = lay.to_one ? e : e >> lg;
    if (slot >= cap) {
      drop(x);
      return false;
    }
    LocalEntry en;
    en.edges = (unsigned long long)(bx + (long long)u * per * C) | (unsigned long long)min(deg - u * per, per) << 44;
    en.orig = og;
    en.row = u == 0 ? x : -1 - x;
    LocalSmem* T = cl.map_shared_rank(&S, lay.to_one ? 0 : (from + e) & ((1 << lg) - 1));
    *reinterpret_cast<int4*>(&T->ent[p][seg + slot]) = *reinterpret_cast<const int4*>(&en);
    return true;
  }
  // Entries of up to N rows a lane (those with x >= 0); all lanes of the warp call, and
  // number their entries with one shared atomic.
  template <int N>
  __device__ __forceinline__ void operator()(const int* x, const long long* bx, const int* deg, const int* og) {
    const int lane = threadIdx.x & 31;
    const int G = 1 << lg, cap = lay.cap(lg), from = first ? 0 : rank;
    const int seg = lay.from_one ? 0 : rank * cap;
    bool single = true;  // every row is one entry
#pragma unroll
    for (int q = 0; q < N; ++q) single = single && (x[q] < 0 || deg[q] <= LOCAL_EDGES);
    if (__all_sync(SS_FULL_MASK, single)) {
      unsigned m[N];
      int at[N], all = 0;
#pragma unroll
      for (int q = 0; q < N; ++q) {
        m[q] = __ballot_sync(SS_FULL_MASK, x[q] >= 0);
        at[q] = all + __popc(m[q] & ((1u << lane) - 1u));
        all += __popc(m[q]);
      }
      int e0 = 0;
      if (lane == 0) e0 = first ? (int)atomicAdd(d.qcount, (unsigned long long)all) : atomicAdd(&mine->nent, all);
      e0 = __shfl_sync(SS_FULL_MASK, e0, 0);
#pragma unroll
      for (int q = 0; q < N; ++q) {
        if (x[q] < 0) continue;
        const int e = e0 + at[q];
        const int slot = lay.to_one ? e : e >> lg;
        if (slot >= cap) {
          drop(x[q]);
          continue;
        }
        LocalEntry en;
        en.edges = (unsigned long long)bx[q] | (unsigned long long)deg[q] << 44;
        en.orig = og[q];
        en.row = x[q];
        LocalSmem* T = cl.map_shared_rank(&S, lay.to_one ? 0 : (from + e) & (G - 1));
        *reinterpret_cast<int4*>(&T->ent[p][seg + slot]) = *reinterpret_cast<const int4*>(&en);
#pragma unroll
        for (int j = 0; j < LOCAL_EDGES; ++j)  // its columns, for the next level
          if (j < deg[q] && !late) asm volatile("prefetch.global.L2 [%0];" ::"l"(d.col + bx[q] + (long long)j * C));
      }
      return;
    }
    int nu[N], total = 0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      nu[q] = 0;
      if (x[q] >= 0) {
        nu[q] = deg[q] > LOCAL_LONG ? (deg[q] + LOCAL_UNIT - 1) / LOCAL_UNIT : (deg[q] + LOCAL_EDGES - 1) / LOCAL_EDGES;
        // a level of more edges than the cluster takes is handed back, so nothing past that is
        // placed (the 160 units of one 163 K hub were 15 us of a Kronecker 22 level)
        if (deg[q] > LOCAL_LONG &&
            atomicAdd(&S.placed[p], (unsigned)min(deg[q], 1 << 17)) + (unsigned)deg[q] > (unsigned)d.local_max_e) {
          drop(x[q]);
          nu[q] = 0;
        }
        total += nu[q];
      }
    }
    int incl = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(SS_FULL_MASK, incl, o);
      if (lane >= o) incl += t;
    }
    const int all = __shfl_sync(SS_FULL_MASK, incl, 31);
    if (all == 0) return;
    int e0 = 0;
    if (lane == 31) e0 = first ? (int)atomicAdd(d.qcount, (unsigned long long)all) : atomicAdd(&mine->nent, all);
    e0 = __shfl_sync(SS_FULL_MASK, e0, 31) + incl - total;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int per = deg[q] > LOCAL_LONG ? LOCAL_UNIT : LOCAL_EDGES;
      if (nu[q] <= LOCAL_LONG / LOCAL_EDGES) {
        for (int u = 0; u < nu[q]; ++u)
          if (!put(x[q], bx[q], deg[q], og[q], per, u, e0 + u, seg, cap, from)) break;
      }
      // the units of a long row, by the whole warp
      unsigned big = __ballot_sync(SS_FULL_MASK, nu[q] > LOCAL_LONG / LOCAL_EDGES);
      while (big) {
        const int src = __ffs(big) - 1;
        big &= big - 1;
        const int bxr = __shfl_sync(SS_FULL_MASK, x[q], src), bdeg = __shfl_sync(SS_FULL_MASK, deg[q], src);
        const int bog = __shfl_sync(SS_FULL_MASK, og[q], src), be = __shfl_sync(SS_FULL_MASK, e0, src);
        const int bn = __shfl_sync(SS_FULL_MASK, nu[q], src);
        const long long bb = __shfl_sync(SS_FULL_MASK, bx[q], src);
        for (int u = lane; u < bn; u += 32)
          if (!put(bxr, bb, bdeg, bog, LOCAL_UNIT, u, be + u, seg, cap, from)) break;
      }
      e0 += nu[q];
    }
  }
};

// atomicMax under a predicate (~0 without it).  Written as a branch, each of a
// thread's claims waited for the one before it at the branch's end: 3,480 cycles for
// four against 1,050 in flight together.
__device__ __forceinline__ unsigned long long claim_if(unsigned long long* p, unsigned long long key, bool on) {
  unsigned long long old;
  asm volatile(
      "{\n\t.reg .pred on;\n\tsetp.ne.s32 on, %3, 0;\n\tmov.b64 %0, -1;\n\t"
      "@on atom.global.max.u64 %0, [%1], %2;\n\t}"
      : "=l"(old)
      : "l"(p), "l"(key), "r"((int)on)
      : "memory");
  return old;
}

// Per-thread counters of a level.
struct LocalSum {
  int nnew = 0;
  unsigned md = 0;
  unsigned long long nd = 0;
};

// Claim up to LOCAL_EDGES neighbours, at b, b + step, ... (n of them) of the row with
// original id og and value fu: every load in flight before a claim, every claim
// before a result, and the discovered rows' data before the first is placed.  All
// lanes of the warp call.
template <int SR, int C>
__device__ __forceinline__ void local_claim(const Dev& d, LocalPlace<C>& place, LocalSum& sum, long long b, int step,
                                            int n, int og, float fu) {
  int v[LOCAL_EDGES];
#pragma unroll
  for (int q = 0; q < LOCAL_EDGES; ++q) v[q] = q < n ? __ldg(d.col + b + (long long)q * step) : -1;
  unsigned long long old[LOCAL_EDGES];
  const unsigned long long key = claim_word(place.k, og);
#pragma unroll
  for (int q = 0; q < LOCAL_EDGES; ++q) old[q] = claim_if(d.claim + v[q], key, v[q] >= 0);
  if (SR == SS_REAL) {  // a neighbour not visited at an earlier level
#pragma unroll
    for (int q = 0; q < LOCAL_EDGES; ++q)
      if ((unsigned)(old[q] >> 32) <= (unsigned)(key >> 32)) atomicAdd(d.psum + v[q], fu);
  }
  // the neighbours' row data, in flight with the claims (of every neighbour: waiting to
  // learn which are new would add a memory latency to the level); in a large level, bound
  // by its accesses and not by their latency, of the new ones alone
  if (place.late) {
#pragma unroll
    for (int q = 0; q < LOCAL_EDGES; ++q)
      if (old[q] != 0ull) v[q] = -1;
  }
  int dv[LOCAL_EDGES], og2[LOCAL_EDGES];
  long long bx[LOCAL_EDGES];
#pragma unroll
  for (int q = 0; q < LOCAL_EDGES; ++q) {
    dv[q] = v[q] >= 0 ? __ldg(d.rdeg + v[q]) : 0;
    bx[q] = v[q] >= 0 ? __ldg(d.cs + v[q] / C) + v[q] % C : 0;
    og2[q] = v[q] >= 0 ? __ldg(d.perm + v[q]) : 0;
  }
  bool any = false;
#pragma unroll
  for (int q = 0; q < LOCAL_EDGES; ++q) {
    if (old[q] != 0ull) v[q] = -1;  // (not discovered here)
    any = any || v[q] >= 0;
  }
  if (!__any_sync(SS_FULL_MASK, any)) return;
  place.template operator()<LOCAL_EDGES>(v, bx, dv, og2);
#pragma unroll
  for (int q = 0; q < LOCAL_EDGES; ++q)
    if (v[q] >= 0) {
      sum.nnew += 1;
      sum.nd += (unsigned long long)dv[q];
      sum.md = max(sum.md, (unsigned)dv[q]);
    }
}

template <int SR, int C>
__global__ void __launch_bounds__(LOCAL_THREADS, 1) k_push_local(Dev d, IterLaunch il, int max_levels,
                                                                 int time_levels) {
  LocalSmem& S = *reinterpret_cast<LocalSmem*>(ss_local_smem);
  // per-level timing (profiling): the first level also carries the launch's entry
  unsigned long long t_prev = time_levels ? global_ns() : 0ull;
  cg::cluster_group cl = cg::this_cluster();
  const int G = (int)cl.num_blocks();  // 8 or 16
  const int lg = 31 - __clz(G);
  const int rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  Ctl* c = d.ctl;
  int k = c->k;
  const int k0 = k;  // first level of this launch (its features came from the decide kernel)
  const int done = c->done;
  unsigned long long nf = c->prev_new, E = c->prev_deg;  // rows and edges of the level-(k-1) frontier
  unsigned long long reached = c->reached, reached_deg = c->reached_deg;
  if (rank == 0)
    for (int i = tid; i < CTL_WORDS; i += LOCAL_THREADS)
      reinterpret_cast<unsigned*>(&S.ctl)[i] = reinterpret_cast<const unsigned*>(c)[i];
  if (tid < 3) S.mine[tid] = LocalPub{0, 0, 0u, 0, 0u, 0u};
  if (tid < 2) S.placed[tid] = 0u;
  if (rank == 0 && tid == 0) *d.qcount = 0ull;  // first entries
  cl.sync();  // every CTA has read the control block, and its counters are reset
  if (done) return;
  bool handback = true;  // (else the run has ended)
  int last = k - 1;      // level of the frontier that the entries hold
  // (the first entries fit: at most nf + E / LOCAL_EDGES, which local_fits bounds by the cluster's capacity)
  LocalLay cur{true, nf + E <= SOLO_DOWN};
  if (!local_fits(d, nf, E)) {  // the decide kernel never sends such a frontier
    if (rank == 0 && tid == 0) {
      S.ctl.error |= 8;
      S.ctl.done = 1;
    }
    handback = false;
    cur = LocalLay{true, true};
    nf = 0;
  }
  // the first entries, from the frontier bitmap (a kernel of its own, listing the rows first,
  // cost each launch 3 us more); the first frontier's bits are cleared, and those of level k-2
  if (handback) {
    const int p1 = (k - 1) & 1;
    LocalPlace<C> place{d, S, cl, &S.mine[0], k, p1, rank, lg, cur, false, true};
    const long long words = ((long long)d.n_pad + 31) / 32;
    unsigned *fbm = d.fb[p1], *fbk = d.fb[k & 1];
    constexpr int AHEAD = 8;  // words in flight per thread
    // a thread takes 1 / 2^sp of a word's bits, so that the rows of a small graph's few words
    // spread over the cluster (the parts of a word lie in one warp)
    const long long threads = (long long)G * LOCAL_THREADS;
    int sp = 0;
    while (sp < 5 && (words << (sp + 1)) <= threads) ++sp;
    const unsigned part = (sp ? (1u << (32 >> sp)) - 1u : ~0u) << ((tid & ((1 << sp) - 1)) * (32 >> sp));
    for (long long t0 = (long long)rank * LOCAL_THREADS + tid; t0 - lane < words << sp; t0 += AHEAD * threads) {
      unsigned bits[AHEAD];
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) {
        const long long w = (t0 + j * threads) >> sp;
        bits[j] = w < words ? __ldcg(fbm + w) : 0u;
        if (w < words) fbk[w] = 0u;
      }
      __syncwarp();  // every lane has read the words that it shares with others before one clears them
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) {
        const long long w = (t0 + j * threads) >> sp;
        if (bits[j]) fbm[w] = 0u;
        bits[j] &= part;
        while (__any_sync(SS_FULL_MASK, bits[j] != 0u)) {
          int u = -1, dv = 0, og = 0;
          long long bx = 0;
          if (bits[j]) {
            u = (int)(w * 32 + __ffs(bits[j]) - 1);
            bits[j] &= bits[j] - 1;
            bx = __ldg(d.cs + u / C) + (u % C);
            dv = __ldg(d.rdeg + u);
            og = __ldg(d.perm + u);
          }
          if (dv == 0) u = -1;  // (an isolated root has no edges)
          place.template operator()<1>(&u, &bx, &dv, &og);
        }
      }
    }
  }
  cl.sync();  // the first entries are in place
  int made = (int)__ldcg(d.qcount);  // entries of the level that rank 0 (or the launch) has made
  bool stopped = !handback;
  bool dropped = false;  // the last level holds rows without room (bits only)
  for (int lev = 0; !stopped; ++lev) {
    const bool solo = cur.to_one;
    const int p1 = (k - 1) & 1, p0 = k & 1;
    if (solo && rank != 0) {  // rank 0 alone: wait for its message
      cl.sync();
      const LocalMsg m = S.msg;
      k = m.k;
      nf = m.nf;
      E = m.E;
      reached = m.reached;
      reached_deg = m.reached_deg;
      cur = LocalLay{true, m.exit != 0};
      last = k - 1;
      made = S.all[last & 1][0].nent;
      if (tid < 3) S.mine[tid] = LocalPub{0, 0, 0u, 0, 0u, 0u};
      if (tid < 2) S.placed[tid] = 0u;
      __syncthreads();
      if (m.exit) {
        handback = m.handback != 0;
        dropped = m.dropped != 0;
        break;
      }
      continue;
    }
    // where the next level is run follows from this one's size, known to all
    const LocalLay nxt{solo, solo || E <= SOLO_DOWN};
    LocalPub* const mine = &S.mine[k % 3];
    if (tid == 0) {  // the next level's counters (last read before the previous level's barrier)
      S.mine[(k + 1) % 3] = LocalPub{0, 0, 0u, 0, 0u, 0u};
      S.placed[p1] = 0u;
    }
    LocalPlace<C> place{d, S, cl, mine, k, p0, rank, lg, nxt, E > (unsigned long long)LOCAL_THREADS * G, false};
    LocalSum sum;
    local_entries(S, cur, made, p1, rank, lg, [&](int at, bool valid) {
      LocalEntry en{0ull, 0, 0};
      if (valid) *reinterpret_cast<int4*>(&en) = *reinterpret_cast<const int4*>(&S.ent[p1][at]);
      const long long b = (long long)(en.edges & ((1ull << 44) - 1ull));
      const int n = (int)(en.edges >> 44);
      const int og = en.orig;
      // the row's visited bit: here and not at its discovery, where the level's barrier would wait for it
      if (valid && en.row >= 0) atomicOr(d.vis + (en.row >> 5), 1u << (en.row & 31));
      float fu = 0.f;
      if (SR == SS_REAL && valid) {  // the row's value: its sum, final since the last barrier
        const int x = en.row;
        fu = __ldcg((lev == 0 ? d.fr : d.psum) + (x < 0 ? -1 - x : x));
        if (lev > 0 && x >= 0) d.fr[x] = fu;
      }
      local_claim<SR, C>(d, place, sum, b, C, n <= LOCAL_EDGES ? n : 0, og, fu);
      unsigned more = __ballot_sync(SS_FULL_MASK, n > LOCAL_EDGES);
      while (more) {  // long rows: the warp takes 32 x LOCAL_EDGES edges at a time
        const int src = __ffs(more) - 1;
        more &= more - 1;
        const long long bl = __shfl_sync(SS_FULL_MASK, b, src);
        const int nl = __shfl_sync(SS_FULL_MASK, n, src);
        const int ol = __shfl_sync(SS_FULL_MASK, og, src);
        const float fl = SR == SS_REAL ? __shfl_sync(SS_FULL_MASK, fu, src) : 0.f;
        for (int j0 = 0; j0 < nl; j0 += 32 * LOCAL_EDGES) {
          const int j = j0 + lane;
          local_claim<SR, C>(d, place, sum, bl + (long long)j * C, 32 * C, j < nl ? (nl - j + 31) / 32 : 0, ol, fl);
        }
      }
    });
    {  // this CTA's counters of the level
      const unsigned nn = __reduce_add_sync(SS_FULL_MASK, (unsigned)sum.nnew);
      const unsigned md = __reduce_max_sync(SS_FULL_MASK, sum.md);
      if (nn) {  // (a warp's 32 low halves of 20 bits, and its high halves, fit 32 bits)
        const unsigned lo = __reduce_add_sync(SS_FULL_MASK, (unsigned)sum.nd & 0xFFFFFu);
        const unsigned hi = __reduce_add_sync(SS_FULL_MASK, (unsigned)(sum.nd >> 20));
        if (lane == 0) {
          atomicAdd(&mine->nnew, (int)nn);
          atomicMax(&mine->md, md);
          atomicAdd(&mine->nd_lo, lo);
          if (hi) atomicAdd(&mine->nd_hi, hi);
        }
      }
    }
    if (SR == SS_REAL && solo) __threadfence();  // the sums are read past L1 after the barrier
    __syncthreads();
    if (!solo && tid < G) cl.map_shared_rank(&S, tid)->all[p0][rank] = *mine;
    if (!solo) cl.sync();  // every claim, sum and entry of level k is in place
    // ---- totals (every warp alike) and the stop decision ----
    const LocalPub pub = lane >= (solo ? 1 : G) ? LocalPub{0, 0, 0u, 0, 0u, 0u} : solo ? *mine : S.all[p0][lane];
    const unsigned tot = __reduce_add_sync(SS_FULL_MASK, (unsigned)pub.nnew);
    const unsigned tm = __reduce_max_sync(SS_FULL_MASK, pub.md);
    dropped = __any_sync(SS_FULL_MASK, pub.drop != 0);
    // (16 CTAs of 16 warps of 2^25 at most)
    const unsigned long long td = (unsigned long long)__reduce_add_sync(SS_FULL_MASK, pub.nd_lo & 0xFFFFFu) +
                                  ((unsigned long long)__reduce_add_sync(SS_FULL_MASK, (pub.nd_lo >> 20)) << 20) +
                                  ((unsigned long long)__reduce_add_sync(SS_FULL_MASK, pub.nd_hi) << 20);
    reached += tot;
    // the same decision advance_level takes on the control block
    const bool stop = tot == 0 || k >= d.n + 1 || reached > d.reach_cap;
    if (rank == 0 && tid == LOCAL_THREADS - 1) {
      advance_level(d, &S.ctl, k, tot, td, E, 0ull, tm, VAR_PUSH_LOCAL);
      if (time_levels && k < d.iter_cap) {  // device-side time of this level
        const unsigned long long t = global_ns();
        d.iters[k].kernel_ns = (int)min(t - t_prev, 2000000000ull);
        t_prev = t;
      }
    }
    reached_deg += td;
    if (rank == 0 && wid == LOCAL_THREADS / 32 - 2 && lane < 7 && k < d.iter_cap) {
      // the totals the next level's selector features come from (computed at exit)
      const unsigned long long v = lane == 0 ? (unsigned long long)tot : lane == 1 ? td
                                 : lane == 2 ? (unsigned long long)tm : lane == 3 ? E
                                 : lane == 4 ? reached : lane == 5 ? reached_deg : nf;
      d.lstat[(size_t)k * SS_LSTAT + lane] = v;
    }
    nf = tot;
    E = td;
    last = k;
    ++k;
    cur = nxt;
    made = __shfl_sync(SS_FULL_MASK, pub.nent, 0);  // (rank 0's)
    handback = !stop;
    stopped = stop || dropped || lev + 1 >= max_levels || !local_fits(d, nf, E);
    const bool wake = solo && !stopped && E > SOLO_UP;  // the others take part again
    if (wake) {  // rank 0's entries, spread as if it had placed them so
      const int n = min(made, LOCAL_ENTRIES);
      // (in rounds of ascending entries: slot e >> lg never passes what has been read)
      for (int j = 0; j < n; j += LOCAL_THREADS) {
        const int e = j + tid;
        LocalEntry en{0ull, 0, 0};
        if (e < n) *reinterpret_cast<int4*>(&en) = *reinterpret_cast<const int4*>(&S.ent[p0][e]);
        __syncthreads();
        if (e < n)
          *reinterpret_cast<int4*>(&cl.map_shared_rank(&S, e & (G - 1))->ent[p0][e >> lg]) =
              *reinterpret_cast<const int4*>(&en);
      }
      cur.to_one = false;
    }
    if (solo && (stopped || wake)) {  // tell the waiting CTAs
      if (tid < G && tid != 0) {
        cl.map_shared_rank(&S, tid)->all[p0][0] = *mine;
        LocalMsg m;
        m.k = k;
        m.exit = stopped ? 1 : 0;
        m.handback = handback ? 1 : 0;
        m.dropped = dropped ? 1 : 0;
        m.nf = nf;
        m.E = E;
        m.reached = reached;
        m.reached_deg = reached_deg;
        cl.map_shared_rank(&S, tid)->msg = m;
      }
      cl.sync();
    }
  }
  // ---- the launch ends: the last frontier's bits (and real values), then the control block ----
  if (rank == 0 && last >= k0) local_features(d, k0, handback ? last : last - 1);
  if (handback) {
    unsigned* fb = d.fb[last & 1];
    local_entries(S, cur, made, last & 1, rank, lg, [&](int at, bool valid) {
      if (!valid) return;
      const int x = S.ent[last & 1][at].row;
      if (x < 0) return;
      atomicOr(fb + (x >> 5), 1u << (x & 31));
      atomicOr(d.vis + (x >> 5), 1u << (x & 31));
      if (SR == SS_REAL && last >= k0) d.fr[x] = __ldcg(d.psum + x);
    });
    if (SR == SS_REAL && dropped) {  // values of the rows without room: every row of the bitmap
      for (long long w = (long long)rank * LOCAL_THREADS + tid; w < (d.n_pad + 31) / 32; w += (long long)G * LOCAL_THREADS)
        for (unsigned bits = __ldcg(fb + w); bits; bits &= bits - 1) {
          const long long x = w * 32 + __ffs(bits) - 1;
          d.fr[x] = __ldcg(d.psum + x);
        }
    }
  }
  cl.sync();  // no CTA leaves while another may still write its shared memory
  if (rank != 0) return;
  if (tid == 0 && SR == SS_REAL) S.ctl.psum_dirty = 1;
  __syncthreads();
  for (int i = tid; i < CTL_WORDS; i += LOCAL_THREADS)
    reinterpret_cast<unsigned*>(c)[i] = reinterpret_cast<const unsigned*>(&S.ctl)[i];
  if (tid == 0 && il.use_cond) cudaGraphSetConditional(il.cond, handback ? 1u : 0u);
}


static int g_local_cluster[64];  // per device: 0 unknown, -1 none fits, else CTAs per cluster

int push_local_cluster_size() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (g_local_cluster[dev] != 0) return g_local_cluster[dev] > 0 ? g_local_cluster[dev] : 0;
  int best = -1;
  for (int G : {SS_LOCAL_CLUSTER_MAX, 8}) {
    auto kern = k_push_local<SS_TROPICAL, 32>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LocalSmem)) !=
        cudaSuccess)
      break;
    if (G > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
      continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G);
    cfg.blockDim = dim3(LOCAL_THREADS);
    cfg.dynamicSmemBytes = sizeof(LocalSmem);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = G;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters >= 1) {
      best = G;
      break;
    }
  }
  cudaGetLastError();  // a refused size is not an error of a later call
  g_local_cluster[dev] = best;
  return best > 0 ? best : 0;
}

template <int SR, int C>
static ss_status launch_push_local_c(const slimsell_graph* h, const Dev& d, const IterLaunch& il,
                                     int max_levels, cudaStream_t st) {
  const int time_levels = h->profiling ? 1 : 0;
  static std::atomic<unsigned long long> configured{0};
  auto kern = k_push_local<SR, C>;
  if (first_on_device(configured)) {
    SS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(LocalSmem)));
    SS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(d.local_cluster);
  cfg.blockDim = dim3(LOCAL_THREADS);
  cfg.dynamicSmemBytes = sizeof(LocalSmem);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = d.local_cluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  SS_CUDA(cudaLaunchKernelEx(&cfg, kern, d, il, max_levels, time_levels));
  return SS_OK;
}

template <int SR>
static ss_status launch_push_local_sr(const slimsell_graph* h, const Dev& d, const IterLaunch& il,
                                      int max_levels, cudaStream_t st) {
  switch (h->C) {
    case 8: return launch_push_local_c<SR, 8>(h, d, il, max_levels, st);
    case 16: return launch_push_local_c<SR, 16>(h, d, il, max_levels, st);
    case 32: return launch_push_local_c<SR, 32>(h, d, il, max_levels, st);
    default: return launch_push_local_c<SR, 64>(h, d, il, max_levels, st);
  }
}

ss_status launch_push_local(const slimsell_graph* h, const Dev& d, int sr, const IterLaunch& il,
                            int max_levels, cudaStream_t st) {
  switch (sr) {
    case SS_TROPICAL: return launch_push_local_sr<SS_TROPICAL>(h, d, il, max_levels, st);
    case SS_REAL: return launch_push_local_sr<SS_REAL>(h, d, il, max_levels, st);
    case SS_BOOLEAN: return launch_push_local_sr<SS_BOOLEAN>(h, d, il, max_levels, st);
    default: return launch_push_local_sr<SS_SELMAX>(h, d, il, max_levels, st);
  }
}

template <int SR, int C>
static ss_status launch_push_c(const slimsell_graph* h, const Dev& d, const IterLaunch& il,
                               cudaStream_t st) {
  // grids follow the graph size: bitmap words for expand/post, possible units for scatter
  const int gw = vertex_grid(h, 32 * PUSH_THREADS);
  const long long units = (long long)h->n_pad + h->nnz / PUSH_UNIT;
  const int gs = (int)std::max(1LL, std::min((long long)8 * h->num_sms, (units + 7) / 8));
  k_push_expand<C><<<gw, PUSH_THREADS, 0, st>>>(d);
  k_push_scatter<SR, C><<<gs, PUSH_THREADS, 0, st>>>(d);
  k_push_post<SR><<<gw, PUSH_THREADS, 0, st>>>(d, il);
  SS_CUDA(cudaGetLastError());
  return SS_OK;
}

template <int SR>
static ss_status launch_push_sr(const slimsell_graph* h, const Dev& d, const IterLaunch& il,
                                cudaStream_t st) {
  switch (h->C) {
    case 8: return launch_push_c<SR, 8>(h, d, il, st);
    case 16: return launch_push_c<SR, 16>(h, d, il, st);
    case 32: return launch_push_c<SR, 32>(h, d, il, st);
    default: return launch_push_c<SR, 64>(h, d, il, st);
  }
}

ss_status launch_push(const slimsell_graph* h, const Dev& d, int sr, const IterLaunch& il,
                      cudaStream_t st) {
  switch (sr) {
    case SS_TROPICAL: return launch_push_sr<SS_TROPICAL>(h, d, il, st);
    case SS_REAL: return launch_push_sr<SS_REAL>(h, d, il, st);
    case SS_BOOLEAN: return launch_push_sr<SS_BOOLEAN>(h, d, il, st);
    default: return launch_push_sr<SS_SELMAX>(h, d, il, st);
  }
}

}  // namespace ss
