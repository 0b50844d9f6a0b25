// Single-source BFS-SpMV on SlimSell (Section III-A semirings, Section III-B
// SlimSell, Section III-C SlimWork, Section III-D SlimChunk, Section II-C DP).
//
// Vertex state lives in the relabelled row space of the layout:
//   claim[r]    level and parent of row r in one 64-bit word (claim_word; 0 while
//               unvisited): the distance vector d with, for the tropical semiring,
//               the vector f itself, and the parents (sel-max p_k, or the DP parent).
//   vis         1-bit image of the visited rows, which SlimWork tests per chunk.
//   fb[k&1]     1-bit image of the frontier f_k (the rows that entered at level k),
//               double-buffered by level parity.  Every semiring's f_{k-1} is zero
//               outside this set, so x_k = A (x) f_{k-1} only needs the semiring
//               value of the neighbours whose bit is set:
//                 tropical  f^u + 1 = k          (f^u = k - 1 on the frontier; rows
//                                                 with non-frontier visited neighbours
//                                                 are visited themselves and keep f^v)
//                 boolean   1
//                 real      fr[u], the path count u carried into the frontier
//                 sel-max   id(u) + 1
//   fr[r]       real-semiring value of row r when it entered the frontier.
//
// Neighbours are stored in descending original id, so the first frontier hit
// of a row (in column order) is its largest-id frontier neighbour: that is the
// sel-max value and, for the other semirings, the DP parent (Section II-C)
// computed on the fly; a separate DP pass after the iterations is also kept.
//
// The bitmap is gathered once per slot.  Random global gathers cost about one
// L1 cycle each, so each block first stages a prefix of the bitmap (the
// degree-sorted hubs, which receive most edges) in shared memory and reads
// the rest through the read-only path.
//
// One warp processes one work item (chunk i, columns [j0, j1)).  Each lane
// loads 16-byte quads of col: a quad is 4 consecutive rows of one column, so
// lane l always meets rows 4*(l mod C/4) .. +3; lanes sharing rows are combined
// with xor-shuffles.  Split chunks (SlimChunk) combine partial rows with
// atomics; the last item of a chunk to arrive runs the post-processing.
#include <algorithm>

#include <cooperative_groups.h>

#include "ss_pull.cuh"

namespace ss {

// Compile-time tunables of the pull kernel (defaults measured best on GB300).
#ifndef SS_PULL_STEP
#define SS_PULL_STEP 4
#endif
#ifndef SS_PULL_STEP_REAL
#define SS_PULL_STEP_REAL 3  // the real semiring also gathers a value per hit
#endif
#ifndef SS_PULL_STEP_SELL
#define SS_PULL_STEP_SELL 2  // Sell-C-sigma loads a value quad beside each column quad
#endif
#ifndef SS_PULL_PREFETCH
#define SS_PULL_PREFETCH 0  // bulk L2 prefetch distance beyond the next step (0: next step only)
#endif

constexpr int PULL_THREADS = SS_PULL_THREADS;  // one block per SM
#ifndef SS_FILTERED_THREADS
#define SS_FILTERED_THREADS 640
#endif
constexpr int FILTERED_THREADS = SS_FILTERED_THREADS;
#ifndef SS_PULL_SHORT_COLS
#define SS_PULL_SHORT_COLS 4
#endif
constexpr int SHORT_COLS = SS_PULL_SHORT_COLS;  // chunks this short go several per warp
// The filtered pull's chunks in groups of C/4 lanes: every unsplit chunk starts in a
// group and goes on in a whole warp once it is still open after GROUP_TRY columns
// with more than GROUP_LEFT left (8 / 32: 314 us for ER 4 M's largest level; leaving
// with more than 8 left 344, trying 4 columns 322).
#ifndef SS_PULL_GROUP_TRY
#define SS_PULL_GROUP_TRY 8
#endif
#ifndef SS_PULL_GROUP_LEFT
#define SS_PULL_GROUP_LEFT 32
#endif
constexpr int GROUP_TRY = SS_PULL_GROUP_TRY;
constexpr int GROUP_LEFT = SS_PULL_GROUP_LEFT;

// int4 col loads in flight per lane (4 slots each).  STOP: in the filtered pass, whose 20 warps
// an SM have 96 registers a thread for them (a level with few hits on Kronecker 22: 181 us with
// the streaming pass's 4, 170 with 8; real 276 with 3, 254 with 6, 269 with 4).
template <int SR, int FMT, bool STOP = false>
__host__ __device__ constexpr int pull_step() {
  if (STOP) return SR == SS_REAL ? 6 : 8;
  return FMT == SS_FORMAT_SELL ? SS_PULL_STEP_SELL : (SR == SS_REAL ? SS_PULL_STEP_REAL : SS_PULL_STEP);
}
// Bits of the semiring's zero, the value of a Sell-C-sigma padding slot.
template <int SR>
__host__ __device__ constexpr int sell_zero_bits() { return SR == SS_TROPICAL ? 0x7f800000 : 0; }

// A Sell-C-sigma quad read: the slots whose value is the semiring's zero are no
// edges (padding, column 0) and become -1, so the scan treats them as SlimSell
// padding; the values stay in v for the real semiring's multiply.
template <int SR>
__device__ __forceinline__ int4 sell_edges(int4 c, int4 v) {
  constexpr int Z = sell_zero_bits<SR>();
  return make_int4(v.x == Z ? -1 : c.x, v.y == Z ? -1 : c.y, v.z == Z ? -1 : c.z, v.w == Z ? -1 : c.w);
}

enum { MODE_FULL = 0, MODE_SLIMWORK = 1, MODE_FILTERED = 3 };

// Real semiring: a level whose frontier's degree sum exceeds nnz / HUB_EDGE_SHARE
// stages the values of the HUB_VALUE_ROWS highest-degree rows (64 KB) in shared
// memory, where most of its value gathers land (the top 16 K rows of a
// Kronecker graph of scale 22 receive 40 % of all edge endpoints).
#ifndef SS_HUB_VALUE_ROWS
#define SS_HUB_VALUE_ROWS 16384
#endif
constexpr int HUB_VALUE_ROWS = SS_HUB_VALUE_ROWS;
constexpr unsigned long long HUB_EDGE_SHARE = 16;

// Ask the TMA unit to pull [p, p + bytes) into L2 ahead of the warp's loads
// (p 16-byte aligned, bytes a positive multiple of 16).
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
  if (bytes == 0) return;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(p), "r"(bytes) : "memory");
}

constexpr int PREFETCH_BYTES = SS_PULL_PREFETCH;  // col bytes prefetched ahead of each warp

__device__ __forceinline__ int4 shfl_int4(int4 v, int src) {
  return make_int4(__shfl_sync(SS_FULL_MASK, v.x, src), __shfl_sync(SS_FULL_MASK, v.y, src),
                   __shfl_sync(SS_FULL_MASK, v.z, src), __shfl_sync(SS_FULL_MASK, v.w, src));
}

// Combine the 4-bit masks of lanes 0 .. C/4-1 into the chunk's bit words (all lanes call).
template <int C>
__device__ __forceinline__ void gather_bits(unsigned nib, int lane, unsigned* lo, unsigned* hi) {
  constexpr int Q = C / 4;
  if (C <= 32) {
    *lo = __reduce_or_sync(SS_FULL_MASK, lane < Q ? nib << (4 * lane) : 0u);
    *hi = 0u;
  } else {
    *lo = __reduce_or_sync(SS_FULL_MASK, lane < 8 ? nib << (4 * lane) : 0u);
    *hi = __reduce_or_sync(SS_FULL_MASK, (lane >= 8 && lane < 16) ? nib << (4 * (lane - 8)) : 0u);
  }
}

struct Counters {
  unsigned long long nw = 0, deg = 0, slots = 0, act = 0;
  unsigned maxdeg = 0;
};

// Per-row result of one item: best = largest original id among frontier
// neighbours (-1 if none) and, for the real semiring, the sum of their values.
struct RowAcc {
  int best[4];
  float sum[4];
};

// Post-process one chunk (the frontier update of Section III-A): new rows are
// the unvisited rows (live: bit r for this lane's row r) whose x_k is non-zero;
// they get a claim word (level k and the parent), a frontier bit and a visited
// bit (vis: the chunk's visited bits before; prev: rows of this chunk that entered
// the frontier earlier in this pass; *added: the new rows' bits).  All lanes call.
//
// GROUPED: the warp holds 32 / Q chunks at once, lanes g*Q .. g*Q+Q-1 owning all
// rows of chunk g (own = this lane's group has a chunk); otherwise lanes 0..Q-1
// own the rows of the warp's one chunk.
template <int SR, int C, bool GROUPED = false>
__device__ __forceinline__ void post_chunk(const Dev& d, int k, int chunk, int lane, unsigned live,
                                           unsigned long long vis, const RowAcc& a, Counters& cnt,
                                           bool own = true, unsigned long long prev = 0ull,
                                           unsigned long long* added = nullptr) {
  constexpr int Q = C / 4;
  const int lq = GROUPED ? lane % Q : lane;
  const bool owner = GROUPED ? own : lane < Q;
  const int R0 = chunk * C + 4 * lq;
  unsigned nib = 0;
  if (owner) {
#pragma unroll
    for (int r = 0; r < 4; ++r)
      // x_k is non-zero exactly where a row has a frontier neighbour (the real
      // semiring's values are positive path counts), so every semiring tests the hit
      if ((live >> r & 1u) && a.best[r] >= 0) nib |= 1u << r;
    if (nib) {
      const int4 dg = *reinterpret_cast<const int4*>(d.rdeg + R0);
      const int D[4] = {dg.x, dg.y, dg.z, dg.w};
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (nib >> r & 1u) {
          d.claim[R0 + r] = claim_word(k, a.best[r]);  // p_k = p_{k-1} + not(p_{k-1}) (.) x_k / DP parent
          if (SR == SS_REAL) d.fr[R0 + r] = a.sum[r];
          cnt.deg += (unsigned long long)D[r];
          cnt.maxdeg = max(cnt.maxdeg, (unsigned)D[r]);
        }
      cnt.nw += __popc(nib);
    }
  }
  unsigned lo, hi;
  if (GROUPED) {  // OR within each group of Q lanes
    lo = (C <= 32 || lq < 8) ? nib << (4 * (lq & 7)) : 0u;
    hi = (C > 32 && lq >= 8) ? nib << (4 * (lq - 8)) : 0u;
#pragma unroll
    for (int o = 1; o < Q; o <<= 1) {
      lo |= __shfl_xor_sync(SS_FULL_MASK, lo, o);
      if (C > 32) hi |= __shfl_xor_sync(SS_FULL_MASK, hi, o);
    }
  } else {
    gather_bits<C>(nib, lane, &lo, &hi);
  }
  if (owner && lq == 0) {
    store_bits<C>(d.fb[k & 1], chunk, lo | (unsigned)prev, hi | (unsigned)(prev >> 32));
    if (lo | hi) store_bits<C>(d.vis, chunk, (unsigned)vis | lo, (unsigned)(vis >> 32) | hi);
  }
  if (added) *added = ((unsigned long long)hi << 32) | lo;
}

// Scan the slots of one quad: record the first frontier hit per row and, for
// the real semiring, add the values of all hits.
// live: bit r set while row r is unvisited.  Visited rows keep their value, so
// the real semiring gathers frontier values for live rows only, and only in a
// branch taken when a live row of the quad was hit (the full passes of the first
// levels see almost no hits).  Values of rows below sf come from the copy staged
// in shared memory (smf), the others from global memory.  (Skipping the bit
// lookups of rows already hit, for the other semirings, measured slower: the
// predicated lookups cost more issue slots than they save.)
//
// Sell-C-sigma (FMT = SS_FORMAT_SELL): the caller has turned the quad's padding
// into -1 (sell_edges), and the real semiring multiplies the gathered value by
// the slot's matrix value v.  The real semiring over SlimSell takes quad_hits
// and gather_step instead, which gather a whole step's values at once.
template <int SR, int FMT>
__device__ __forceinline__ void scan_quad(const Dev& d, const unsigned* sm, int sbits,
                                          const unsigned* gbm, int4 c, int4 v, int first[4], float sum[4],
                                          unsigned live, const float* smf, int sf) {
  const int cc[4] = {c.x, c.y, c.z, c.w};
  const int vv[4] = {v.x, v.y, v.z, v.w};
  unsigned hit[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) hit[r] = frontier_bit(sm, sbits, gbm, cc[r]);
#pragma unroll
  for (int r = 0; r < 4; ++r) first[r] = (hit[r] && first[r] < 0) ? cc[r] : first[r];
  if (SR == SS_REAL) {
    const unsigned m = (hit[0] | (hit[1] << 1) | (hit[2] << 2) | (hit[3] << 3)) & live;
    if (m) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (m >> r & 1u) {
          const float x = (cc[r] < sf) ? smf[cc[r]] : __ldg(d.fr + cc[r]);
          sum[r] += (FMT == SS_FORMAT_SELL) ? __int_as_float(vv[r]) * x : x;
        }
    }
  }
}


// Real semiring, SlimSell: the frontier hits of one quad (bit r for row r) and
// the first-hit update; the value gathers follow for the whole step at once.
__device__ __forceinline__ unsigned quad_hits(const unsigned* sm, int sbits, const unsigned* gbm, int4 c,
                                              int first[4]) {
  const int cc[4] = {c.x, c.y, c.z, c.w};
  unsigned m = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const unsigned h = frontier_bit(sm, sbits, gbm, cc[r]);
    first[r] = (h && first[r] < 0) ? cc[r] : first[r];
    m |= h << r;
  }
  return m;
}

// Gather and add the values of every live hit of a step's U quads: all loads are
// issued before the first add, so a warp waits once per step, not once per quad
// (Kronecker 22 hub level: 322 -> 278 us; the gathers are latency-bound, and
// staging more hub rows as 8- or 16-bit counts measured no faster).
template <int U, bool SHARED = false>
__device__ __forceinline__ void gather_step(const Dev& d, const int4* c, const unsigned* mm, float sum[4],
                                            const float* smf, int sf) {
  unsigned any = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) any |= mm[u];
  if (!any) return;
  float x[U][4];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int cc[4] = {c[u].x, c[u].y, c[u].z, c[u].w};
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float v = 0.f;
      if (mm[u] >> r & 1u)
        v = (cc[r] < sf) ? smf[cc[r]] : SHARED ? __ldcg(d.fr + cc[r]) : __ldg(d.fr + cc[r]);
      x[u][r] = v;
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int r = 0; r < 4; ++r) sum[r] += x[u][r];
}


// The frontier bitmap as a block reads it: words of the staged prefix (sbits bits)
// from shared memory, the rest from global memory; real semiring on hub levels:
// the values of the rows below sf from shared memory too.
struct Staged {
  const unsigned* sm;
  const float* smf;
  int sbits, sf;
};

// Stage the prefix of f_{k-1}'s bitmap gbm with asynchronous 16-byte copies (all
// threads of the block call; the copies run until stage_wait).
template <int SR>
__device__ __forceinline__ Staged stage_frontier(const Dev& d, const unsigned* gbm) {
  const int pv = d.ctl->prev_variant;
  const bool light = (pv == VAR_FULL || pv == VAR_SLIMWORK || pv == VAR_FILTERED) &&
                     d.ctl->prev_slots < STAGE_MIN_SLOTS;
  const int sw_all = light ? 0 : d.smem_words;
  // real semiring on a level whose frontier carries a large share of the edges
  // (the hub level of a skewed graph): the last sf words of the staging area
  // hold the values fr of the sf highest-degree rows instead of bitmap words
  const bool hub = SR == SS_REAL && (unsigned long long)d.ctl->prev_deg * HUB_EDGE_SHARE >
                                        (unsigned long long)d.nnz;
  const int sf = hub ? min(HUB_VALUE_ROWS, (sw_all >> 1) & ~3) : 0;
  const int sw = sw_all - sf;  // bitmap words staged (a multiple of 4)
  if (threadIdx.x < SMEM_GUARD) ss_smem_bits[threadIdx.x] = 0u;
  const unsigned sbase = stage_words(gbm, sw);
  const unsigned fbase = sbase + 4u * (unsigned)sw;
  for (int i = threadIdx.x; i < (sf >> 2); i += blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(fbase + 16u * (unsigned)i),
                 "l"(reinterpret_cast<const int4*>(d.fr) + i)
                 : "memory");
  Staged s;
  s.sm = ss_smem_bits + SMEM_GUARD;
  s.smf = reinterpret_cast<const float*>(s.sm + sw);
  s.sbits = sw * 32;
  s.sf = sf;
  return s;
}
struct __align__(8) ItemCache {
  int chunk, y, z, w;
  long long start;
};

// The items of a warp's batch that take a whole warp each (todo: their lanes, lane s holding
// item s).  STOP (the filtered pass): rows that are visited or, but for the real semiring,
// hit load nothing more; counted: items that are counted as active already; found: rows of
// this lane's item that entered the frontier earlier in this pass.
template <int SR, int C, int FMT, bool SHARED, bool STOP>
__device__ __forceinline__ void pull_whole(const Dev& d, int k, const unsigned* gbm, const Staged& sg, unsigned todo,
                                           const int4& my_item, long long my_start, unsigned long long my_vis,
                                           Counters& cnt, unsigned counted = 0u, unsigned long long found = 0ull) {
  constexpr int PULL_STEP = pull_step<SR, FMT, STOP>();
  constexpr int Q = C / 4;
  const int* colp = (FMT == SS_FORMAT_SELL) ? d.scol : d.col;
  const int lane = threadIdx.x & 31;
  const unsigned* sm = sg.sm;
  const float* smf = sg.smf;
  const int sbits = sg.sbits, sf = sg.sf;
  while (todo) {
    const int src = __ffs(todo) - 1;
    todo &= todo - 1;
    const int4 item = shfl_int4(my_item, src);
    const long long start = __shfl_sync(SS_FULL_MASK, my_start, src);
    const int chunk = item.x;
    // L2 prefetch: the head of this item beyond the first step, and of the next item
    if (lane == src) {
      const unsigned bytes = (unsigned)(item.z - item.y) * C * 4u;
      if (bytes > 2048u)
        prefetch_l2(colp + start + 512, min(bytes - 2048u, (unsigned)PREFETCH_BYTES));
    }
    if (todo) {
      const int nxt = __ffs(todo) - 1;
      if (lane == nxt) {
        const unsigned bytes = (unsigned)(my_item.z - my_item.y) * C * 4u;
        prefetch_l2(colp + my_start, min(bytes, (unsigned)PREFETCH_BYTES));
      }
    }
    // this lane's unvisited rows (only this chunk's post changes them)
    const unsigned long long vis = __shfl_sync(SS_FULL_MASK, my_vis, src);
    const unsigned live = ~(unsigned)(vis >> (4 * (lane % Q))) & 0xFu;
    int first[4] = {-1, -1, -1, -1};
    float sum[4] = {0.f, 0.f, 0.f, 0.f};
    bool need = live != 0u;  // (STOP)
    const int nq = (item.z - item.y) * Q;
    const int4* base = reinterpret_cast<const int4*>(colp + start);
    const int4* vbase = reinterpret_cast<const int4*>(d.sval + start);  // (Sell only)
    for (int q0 = 0; q0 < nq; q0 += 32 * PULL_STEP) {
      if (STOP) {
        if (!__any_sync(SS_FULL_MASK, need)) break;
        if (!need) continue;
      }
      // keep the prefetch PREFETCH_BYTES ahead inside long items (one lane issues it)
      if (lane == 0) {
        const long long ahead = (long long)(q0 + 32 * PULL_STEP) * 16 + PREFETCH_BYTES;
        const long long total = (long long)nq * 16;
        if (ahead < total) {
          prefetch_l2(reinterpret_cast<const char*>(base) + ahead,
                      (unsigned)min(total - ahead, (long long)(32 * PULL_STEP * 16)));
          if (FMT == SS_FORMAT_SELL)
            prefetch_l2(reinterpret_cast<const char*>(vbase) + ahead,
                        (unsigned)min(total - ahead, (long long)(32 * PULL_STEP * 16)));
        }
      }
      int4 c[PULL_STEP], v[PULL_STEP];
#pragma unroll
      for (int u = 0; u < PULL_STEP; ++u) {
        const int q = q0 + lane + 32 * u;
        c[u] = (q < nq) ? ld_stream(base + q) : make_int4(-1, -1, -1, -1);
        if (STOP && q < nq) cnt.slots += 4;
        if (FMT == SS_FORMAT_SELL) {
          const int4 vq = (q < nq) ? ld_stream(vbase + q) : make_int4(0, 0, 0, 0);
          c[u] = sell_edges<SR>(c[u], vq);
          v[u] = SR == SS_REAL ? vq : make_int4(0, 0, 0, 0);
        } else {
          v[u] = make_int4(0, 0, 0, 0);
        }
      }
      if constexpr (SR == SS_REAL && FMT == SS_FORMAT_SLIMSELL) {
        unsigned mm[PULL_STEP];
#pragma unroll
        for (int u = 0; u < PULL_STEP; ++u)
          mm[u] = (q0 + 32 * u < nq) ? quad_hits(sm, sbits, gbm, c[u], first) & live : 0u;
        gather_step<PULL_STEP, SHARED>(d, c, mm, sum, smf, sf);
      } else {
#pragma unroll
        for (int u = 0; u < PULL_STEP; ++u)  // (q0 + 32 u < nq is warp-uniform)
          if (q0 + 32 * u < nq) scan_quad<SR, FMT>(d, sm, sbits, gbm, c[u], v[u], first, sum, live, smf, sf);
      }
      if (STOP) {  // a row is done once visited or (not real) hit
        need = false;
#pragma unroll
        for (int r = 0; r < 4; ++r) need |= (live >> r & 1u) && (SR == SS_REAL || first[r] < 0);
      }
    }
    if (!STOP && lane == 0) cnt.slots += (unsigned long long)(item.z - item.y) * C;
    // the largest original id among this lane's first hits of unvisited rows
    RowAcc acc;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      acc.best[r] = (first[r] >= 0 && (live >> r & 1u)) ? __ldg(d.perm + first[r]) : -1;
      acc.sum[r] = sum[r];
    }
    // (a non-zero real sum implies a hit on a live row of the same lane)
    const bool any_hit = (acc.best[0] >= 0) | (acc.best[1] >= 0) | (acc.best[2] >= 0) |
                         (acc.best[3] >= 0);
    if (__any_sync(SS_FULL_MASK, any_hit)) {  // lanes with equal lane mod Q share rows
#pragma unroll
      for (int off = Q; off < 32; off <<= 1)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          acc.best[r] = max(acc.best[r], __shfl_xor_sync(SS_FULL_MASK, acc.best[r], off));
          if (SR == SS_REAL) acc.sum[r] += __shfl_xor_sync(SS_FULL_MASK, acc.sum[r], off);
        }
    }
    if (item.w >= 0) {  // SlimChunk: combine partial rows, the last arriving item post-processes
      const size_t xo = (size_t)item.w * C + 4 * lane;
      if (lane < Q) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if (acc.best[r] >= 0) atomicMax(d.xpar + xo + r, acc.best[r]);
          if (SR == SS_REAL && acc.sum[r] != 0.0f) atomicAdd(d.xacc + xo + r, acc.sum[r]);
        }
        __threadfence();
      }
      __syncwarp();
      int last = 0;
      if (lane == 0) {
        const unsigned old = atomicAdd(d.arrive + item.w, 1u);
        last = (old == (unsigned)d.split_n[item.w] - 1u);
      }
      last = __shfl_sync(SS_FULL_MASK, last, 0);
      if (!last) continue;
      __threadfence();
      if (lane < Q) {
        // one 16-byte read and reset per array (xo is a multiple of 4 and the
        // scratch 16-byte aligned); the per-row scalar form of this rarely run
        // block made the whole real-semiring kernel 20-25 % slower on GB300
        const int4 b4 = __ldcg(reinterpret_cast<const int4*>(d.xpar + xo));
        *reinterpret_cast<int4*>(d.xpar + xo) = make_int4(-1, -1, -1, -1);
        acc.best[0] = b4.x; acc.best[1] = b4.y; acc.best[2] = b4.z; acc.best[3] = b4.w;
        if (SR == SS_REAL) {
          const float4 s4 = __ldcg(reinterpret_cast<const float4*>(d.xacc + xo));
          *reinterpret_cast<float4*>(d.xacc + xo) = make_float4(0.f, 0.f, 0.f, 0.f);
          acc.sum[0] = s4.x; acc.sum[1] = s4.y; acc.sum[2] = s4.z; acc.sum[3] = s4.w;
        }
      }
      if (lane == 0) d.arrive[item.w] = 0u;
    }
    if (lane == 0 && !(STOP && (counted >> src & 1u))) cnt.act += 1;
    post_chunk<SR, C>(d, k, chunk, lane, live, vis, acc, cnt, true, STOP ? __shfl_sync(SS_FULL_MASK, found, src) : 0ull);
  }
}

// Warp wid of nw walks its items wid, wid + nw, ... of level k (the item list is
// ordered for such an assignment): it reads the descriptors and visited bits of 32
// of them at once (one per lane) and processes the active ones.  full: every chunk
// is active.  SHARED: other SMs have written the bitmaps and values since this
// kernel began, so those are read past L1 (and the whole bitmap is staged); cache:
// the threads' item descriptors in shared memory (at most one batch), filled by the
// first level.  STOP: see pull_whole.
template <int SR, int C, int FMT, bool SHARED, bool STOP = false>
__device__ __forceinline__ void pull_items(const Dev& d, int k, bool full, const unsigned* gbm, const Staged& sg,
                                           int wid, int nw, Counters& cnt, ItemCache* cache = nullptr,
                                           bool fill = false) {
  constexpr int Q = C / 4;
  constexpr unsigned long long ALL_ROWS = C == 64 ? ~0ull : (1ull << C) - 1ull;
  const int* colp = (FMT == SS_FORMAT_SELL) ? d.scol : d.col;
  const int lane = threadIdx.x & 31;
  const unsigned* sm = sg.sm;
  const float* smf = sg.smf;
  const int sbits = sg.sbits, sf = sg.sf;
  for (long long b0 = wid; b0 < d.n_items; b0 += 32LL * nw) {
    const long long my_it = b0 + (long long)lane * nw;
    int4 my_item = make_int4(0, 0, 0, -1);
    long long my_start = 0;
    unsigned long long my_vis = ALL_ROWS;  // the chunk's visited rows
    bool active = false;
    if (my_it < d.n_items) {
      if (SHARED && cache && !fill) {
        const ItemCache ic = cache[threadIdx.x];
        my_item = make_int4(ic.chunk, ic.y, ic.z, ic.w);
        my_start = ic.start;
      } else {
        my_item = d.items[my_it];
        my_start = d.cs[my_item.x] + (long long)my_item.y * C;
        if (SHARED && cache)
          cache[threadIdx.x] = ItemCache{my_item.x, my_item.y, my_item.z, my_item.w, my_start};
      }
      my_vis = chunk_bits<C, SHARED>(d.vis, my_item.x);
      const unsigned long long old = chunk_bits<C, SHARED>(d.fb[k & 1], my_item.x);  // in flight with vis
      active = full || my_vis != ALL_ROWS;
      // a finished chunk (SlimWork) adds no row: f_k is zero there, so what
      // f_{k-2} left in the parity buffer is cleared
      if (!active && my_item.y == 0 && old != 0ull) store_bits<C>(d.fb[k & 1], my_item.x, 0u, 0u);
    }
    unsigned todo = __ballot_sync(SS_FULL_MASK, active);
    // short whole chunks (at most SHORT_COLS columns, about half of all chunks of a
    // skewed graph) go 32 / Q at a time, one group of Q lanes each
    unsigned shortm = __ballot_sync(SS_FULL_MASK, active && my_item.w < 0 &&
                                                      my_item.z - my_item.y <= SHORT_COLS);
    todo &= ~shortm;
    while (shortm) {
      constexpr int GROUPS = 32 / Q;
      int mysrc = -1;
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) {
        const int sidx = shortm ? __ffs(shortm) - 1 : -1;
        if (lane / Q == g) mysrc = sidx;
        shortm &= shortm - 1;
      }
      const bool own = mysrc >= 0;
      const int sl = own ? mysrc : 0;
      const int4 item = make_int4(__shfl_sync(SS_FULL_MASK, my_item.x, sl),
                                  __shfl_sync(SS_FULL_MASK, my_item.y, sl),
                                  __shfl_sync(SS_FULL_MASK, my_item.z, sl), -1);
      const long long start = __shfl_sync(SS_FULL_MASK, my_start, sl);
      const int lq = lane % Q;
      const int ncols = own ? item.z - item.y : 0;
      const int chunk = item.x;
      const unsigned long long vis = __shfl_sync(SS_FULL_MASK, my_vis, sl);
      const unsigned live = own ? ~(unsigned)(vis >> (4 * lq)) & 0xFu : 0u;
      int first[4] = {-1, -1, -1, -1};
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
      const int4* base = reinterpret_cast<const int4*>(colp + start) + lq;
      const int4* vbase = reinterpret_cast<const int4*>(d.sval + start) + lq;  // (Sell only)
      int4 c[SHORT_COLS], v[SHORT_COLS];
#pragma unroll
      for (int u = 0; u < SHORT_COLS; ++u) {
        c[u] = (u < ncols) ? ld_stream(base + u * Q) : make_int4(-1, -1, -1, -1);
        if (FMT == SS_FORMAT_SELL) {
          const int4 vq = (u < ncols) ? ld_stream(vbase + u * Q) : make_int4(0, 0, 0, 0);
          c[u] = sell_edges<SR>(c[u], vq);
          v[u] = SR == SS_REAL ? vq : make_int4(0, 0, 0, 0);
        } else {
          v[u] = make_int4(0, 0, 0, 0);
        }
      }
      if constexpr (SR == SS_REAL && FMT == SS_FORMAT_SLIMSELL) {
        unsigned mm[SHORT_COLS];
#pragma unroll
        for (int u = 0; u < SHORT_COLS; ++u)
          mm[u] = (u < ncols) ? quad_hits(sm, sbits, gbm, c[u], first) & live : 0u;
        gather_step<SHORT_COLS, SHARED>(d, c, mm, sum, smf, sf);
      } else {
#pragma unroll
        for (int u = 0; u < SHORT_COLS; ++u)
          if (u < ncols) scan_quad<SR, FMT>(d, sm, sbits, gbm, c[u], v[u], first, sum, live, smf, sf);
      }
      if (own && lq == 0) {
        cnt.act += 1;
        cnt.slots += (unsigned long long)ncols * C;
      }
      RowAcc acc;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        acc.best[r] = (first[r] >= 0 && (live >> r & 1u)) ? __ldg(d.perm + first[r]) : -1;
        acc.sum[r] = sum[r];
      }
      post_chunk<SR, C, true>(d, k, chunk, lane, live, vis, acc, cnt, own);
    }
    pull_whole<SR, C, FMT, SHARED, STOP>(d, k, gbm, sg, todo, my_item, my_start, my_vis, cnt);
  }
}

// The first level, whose frontier is the root alone: x_1 is non-zero exactly in the
// rows of the slots that hold the root, so the pass streams the whole column array
// against one row number, eight 16-byte quads in flight per lane, with no item walk, no
// bitmap and no lookup, and is bound by HBM.  A slot that holds the root (one per
// neighbour) finds its chunk by bisection; only that row's chunk is SlimWork-skipped
// (and its slots not counted) when its rows are all visited.  Not for the real semiring,
// where a repeated edge counts twice.  From ROOT_MIN_SLOTS slots on: below, the level
// is launch and latency either way.  Level 1 of Kronecker 22: 128 us to 96 (533 MB), of
// Kronecker 24 520 to 332 (2.2 GB); a whole run of Kronecker 18 178 to 160.
#ifndef SS_ROOT_MIN_SLOTS
#define SS_ROOT_MIN_SLOTS (4LL << 20)
#endif
constexpr long long ROOT_MIN_SLOTS = SS_ROOT_MIN_SLOTS;
template <int C>
__device__ __forceinline__ void pull_root(const Dev& d, bool full, Counters& cnt) {
  constexpr int U = 8;
  const int root_row = d.ctl->root_row;
  const int root = __ldg(d.perm + root_row);
  const int lane = threadIdx.x & 31;
  const long long nq = d.total_slots >> 2;
  const long long warps = (long long)gridDim.x * (PULL_THREADS / 32);
  const int4* col = reinterpret_cast<const int4*>(d.col);
  for (long long q0 = ((long long)blockIdx.x * (PULL_THREADS / 32) + (threadIdx.x >> 5)) * (32 * U); q0 < nq;
       q0 += warps * (32 * U)) {
    int4 c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const long long q = q0 + lane + 32 * u;
      c[u] = q < nq ? ld_stream(col + q) : make_int4(-1, -1, -1, -1);
    }
    bool any = false;
#pragma unroll
    for (int u = 0; u < U; ++u)
      any = any || c[u].x == root_row || c[u].y == root_row || c[u].z == root_row || c[u].w == root_row;
    if (!any) continue;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int cc[4] = {c[u].x, c[u].y, c[u].z, c[u].w};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if (cc[r] != root_row) continue;
        const long long slot = 4 * (q0 + lane + 32 * u) + r;
        int lo = 0, hi = d.n_c - 1;  // the last chunk that starts at or before the slot
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (__ldg(d.cs + mid) <= slot) lo = mid;
          else hi = mid - 1;
        }
        const long long row = (long long)lo * C + (slot - __ldg(d.cs + lo)) % C;
        const unsigned bit = 1u << (row & 31);
        if (atomicOr(d.vis + (row >> 5), bit) & bit) continue;  // the root, or a repeated edge
        const int dg = __ldg(d.rdeg + row);
        d.claim[row] = claim_word(1, root);
        atomicOr(d.fb[1] + (row >> 5), bit);
        cnt.nw += 1;
        cnt.deg += (unsigned long long)dg;
        cnt.maxdeg = max(cnt.maxdeg, (unsigned)dg);
      }
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    cnt.slots = (unsigned long long)d.total_slots;
    cnt.act = (unsigned long long)d.n_busy;
    const int rc = root_row / C;  // its chunk is finished when the root is its only real row
    if (!full && d.cl[rc] > 0 && d.n - rc * C == 1) {
      cnt.slots -= (unsigned long long)d.cl[rc] * C;
      cnt.act -= 1;
    }
  }
}

// One frontier expansion x_k = A (x)_S f_{k-1} with fused post-processing.
template <int SR, int C, int MODE, int FMT>
__global__ void __launch_bounds__(PULL_THREADS, 1) k_pull(Dev d, int variant,
                                                          cudaGraphConditionalHandle cond,
                                                          int use_cond) {
  if (d.ctl->done) return;
  const int k = d.ctl->k;
  Counters cnt;
  if (FMT == SS_FORMAT_SLIMSELL && SR != SS_REAL && k == 1 && d.total_slots >= ROOT_MIN_SLOTS) {
    pull_root<C>(d, MODE == MODE_FULL, cnt);
    finish_iteration_block<PULL_THREADS>(d, cnt.nw, cnt.deg, cnt.slots, cnt.act, cnt.maxdeg,
                                         IterLaunch{variant, cond, use_cond});
    return;
  }
  const unsigned* gbm = d.fb[(k - 1) & 1];
  const Staged sg = stage_frontier<SR>(d, gbm);
  stage_wait();
  pull_items<SR, C, FMT, false>(d, k, MODE == MODE_FULL, gbm, sg,
                                (int)(blockIdx.x * (PULL_THREADS / 32) + (threadIdx.x >> 5)),
                                (int)(gridDim.x * (PULL_THREADS / 32)), cnt);
  finish_iteration_block<PULL_THREADS>(d, cnt.nw, cnt.deg, cnt.slots, cnt.act, cnt.maxdeg,
                                       IterLaunch{variant, cond, use_cond});
}

// The visited-filtered pull: as k_pull, but only unvisited rows are computed and
// (but for the real semiring) a row stops at its first frontier neighbour.
//
// Where the frontier's rows hold a good share of all edges (frontier_hits_soon), most rows
// stop within their first columns, so what a pass costs is not the stream but the
// latency chain of each chunk (descriptor, columns, bits, parent, row data).  There
// chunks start in groups of C/4 lanes (32 / (C/4) at a time, GSTEP columns a step, each
// group taking its next chunk on its own), and the next loads are issued before the
// finished chunks are post-processed; only long rests and split items take a whole warp.
// Reading 16 columns at once with one chunk per warp took 64 us on Kronecker 22's level
// after the hubs and 301 us on ER 4 M's largest; this takes 48 and 158 (GSTEP 4: 248 where
// GSTEP 2 took 230; without leaving out the lookups of rows already hit 314).  Elsewhere,
// and for the real semiring, which needs whole sums, the columns are streamed as in
// k_pull: in groups, levels with few hits took 44 us on ER 1 M and 186 on Kronecker 22, and
// 37 and 170 so.  640 threads, for the registers (768: 246 at GSTEP 4; 1024 spills).
// The levels with many hits.
template <int SR, int C>
__device__ __forceinline__ void pull_groups(const Dev& d, int k, const unsigned* gbm, const Staged& sg, int wid, int nw,
                                            Counters& cnt) {
  constexpr int FMT = SS_FORMAT_SLIMSELL;
  constexpr int Q = C / 4;
  constexpr unsigned long long ALL_ROWS = C == 64 ? ~0ull : (1ull << C) - 1ull;
  const int* colp = d.col;
  const int lane = threadIdx.x & 31;
  for (long long b0 = wid; b0 < d.n_items; b0 += 32LL * nw) {
    const long long my_it = b0 + (long long)lane * nw;
    int4 my_item = make_int4(0, 0, 0, -1);
    long long my_start = 0;
    unsigned long long my_vis = ALL_ROWS;  // the chunk's visited rows
    bool active = false;
    if (my_it < d.n_items) {
      my_item = d.items[my_it];
      my_vis = chunk_bits<C>(d.vis, my_item.x);
      my_start = d.cs[my_item.x] + (long long)my_item.y * C;
      const unsigned long long old = chunk_bits<C>(d.fb[k & 1], my_item.x);  // in flight with vis
      active = my_vis != ALL_ROWS;
      // a finished chunk (SlimWork) adds no row: f_k is zero there, so what
      // f_{k-2} left in the parity buffer is cleared
      if (!active && my_item.y == 0 && old != 0ull) store_bits<C>(d.fb[k & 1], my_item.x, 0u, 0u);
    }
    unsigned todo = __ballot_sync(SS_FULL_MASK, active);
    // unsplit chunks in groups of Q lanes.  Each group works through its own
    // chunk GSTEP columns at a time and takes the next one when it is done; the loads
    // of the next step are issued before the finished chunks are post-processed.
    unsigned long long my_new = 0ull;  // rows of this lane's item that the groups have found
    const unsigned grouped = __ballot_sync(SS_FULL_MASK, active && my_item.w < 0);
    {
      constexpr int GROUPS = 32 / Q;
      constexpr int GSTEP = 2;
      const int lq = lane % Q;
      unsigned gm = grouped;
      todo &= ~gm;
      int src = -1, chunk = 0, rem = 0;  // this group's item (its lane), chunk and columns left
      unsigned live = 0;                 // this lane's unvisited rows of it
      unsigned long long vis = 0ull;     // its visited rows
      const int4* cp = nullptr;
      int first[4];
      float none[4] = {0.f, 0.f, 0.f, 0.f};  // (no sums but for the real semiring)
      int4 c[GSTEP];
      // groups that want an item take the next ones; their first step is loaded
      auto take = [&](bool want) {
        const unsigned wm = __ballot_sync(SS_FULL_MASK, want);
        int got = -1;
#pragma unroll
        for (int g = 0; g < GROUPS; ++g)
          if (wm >> (g * Q) & 1u) {
            const int nxt = gm ? __ffs(gm) - 1 : -1;
            gm &= gm - 1;
            if (lane / Q == g) got = nxt;
          }
        const int sl = got >= 0 ? got : 0;
        const int nchunk = __shfl_sync(SS_FULL_MASK, my_item.x, sl);
        const int ncols = __shfl_sync(SS_FULL_MASK, my_item.z, sl) - __shfl_sync(SS_FULL_MASK, my_item.y, sl);
        const long long start = __shfl_sync(SS_FULL_MASK, my_start, sl);
        const unsigned long long nvis = __shfl_sync(SS_FULL_MASK, my_vis, sl);
        if (want) {
          src = got;
          rem = got >= 0 ? ncols : 0;
          chunk = nchunk;
          vis = nvis;
          live = got >= 0 ? ~(unsigned)(nvis >> (4 * lq)) & 0xFu : 0u;
          cp = reinterpret_cast<const int4*>(colp + start) + lq;
          if (got >= 0 && lq == 0) cnt.act += 1;
#pragma unroll
          for (int r = 0; r < 4; ++r) first[r] = -1;
        }
      };
      auto load = [&]() {
        unsigned open = live;
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (first[r] >= 0) open &= ~(1u << r);
        const int n = open ? rem : 0;
        cnt.slots += 4ull * (unsigned)max(0, min(n, GSTEP));
#pragma unroll
        for (int u = 0; u < GSTEP; ++u) c[u] = (u < n) ? ld_stream(cp + u * Q) : make_int4(-1, -1, -1, -1);
      };
      if (gm) {
        take(true);
        load();
      }
      while (__any_sync(SS_FULL_MASK, src >= 0)) {
        // rows hit in an earlier step (or visited) look nothing up: past the staged
        // prefix a lookup is a memory gather
        bool shut[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) shut[r] = first[r] >= 0 || !(live >> r & 1u);
#pragma unroll
        for (int u = 0; u < GSTEP; ++u) {
          const int4 q = make_int4(shut[0] ? -1 : c[u].x, shut[1] ? -1 : c[u].y, shut[2] ? -1 : c[u].z,
                                   shut[3] ? -1 : c[u].w);
          scan_quad<SR, FMT>(d, sg.sm, sg.sbits, gbm, q, make_int4(0, 0, 0, 0), first, none, live, sg.smf, sg.sf);
        }
        rem -= GSTEP;
        cp += GSTEP * Q;
        unsigned open = 0;  // done once every row is visited or hit
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if ((live >> r & 1u) && first[r] < 0) open = 1;
#pragma unroll
        for (int o = 1; o < Q; o <<= 1) open |= __shfl_xor_sync(SS_FULL_MASK, open, o);
        const bool fin = src >= 0 && (rem <= 0 || !open);
        // a long rest goes to the whole warp (from this column on)
        const int used = __shfl_sync(SS_FULL_MASK, my_item.z, max(src, 0)) -
                         __shfl_sync(SS_FULL_MASK, my_item.y, max(src, 0)) - rem;
        const bool leave = src >= 0 && !fin && used >= GROUP_TRY && rem > GROUP_LEFT;
        const bool out = fin || leave;
        if (__any_sync(SS_FULL_MASK, out)) {
          const int ochunk = chunk, osrc = src, orem = rem;
          const unsigned olive = live;
          const unsigned long long ovis = vis;
          RowAcc acc;
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            acc.best[r] = (out && first[r] >= 0 && (live >> r & 1u)) ? first[r] : -1;
            acc.sum[r] = 0.f;
          }
          take(out);
          load();
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (acc.best[r] >= 0) acc.best[r] = __ldg(d.perm + acc.best[r]);
          unsigned long long added;
          post_chunk<SR, C, true>(d, k, ochunk, lane, olive, ovis, acc, cnt, out, 0ull, &added);
          // hand the left chunks over: lane s holds item s
#pragma unroll
          for (int g = 0; g < GROUPS; ++g) {
            const int s = __shfl_sync(SS_FULL_MASK, leave ? osrc : -1, g * Q);
            const int left = __shfl_sync(SS_FULL_MASK, orem, g * Q);
            const unsigned long long nb = __shfl_sync(SS_FULL_MASK, added, g * Q);
            if (s >= 0) {
              todo |= 1u << s;
              if (lane == s) {
                const int y = my_item.z - left;
                my_start += (long long)(y - my_item.y) * C;
                my_item.y = y;
                my_new = nb;
                my_vis |= nb;
              }
            }
          }
        } else {
          load();
        }
      }
    }
    __syncwarp();  // a left chunk's bits, stored by its group's first lane, are stored again by lane 0
    pull_whole<SR, C, FMT, false, true>(d, k, gbm, sg, todo, my_item, my_start, my_vis, cnt, grouped, my_new);
  }
}

template <int SR, int C>
__global__ void __launch_bounds__(FILTERED_THREADS, 1) k_pull_filtered(Dev d, int variant,
                                                                       cudaGraphConditionalHandle cond,
                                                                       int use_cond) {
  if (d.ctl->done) return;
  const int k = d.ctl->k;
  const unsigned* gbm = d.fb[(k - 1) & 1];
  const Staged sg = stage_frontier<SR>(d, gbm);
  const bool many_hits = frontier_hits_soon(d, d.ctl);
  stage_wait();
  const int wid = blockIdx.x * (FILTERED_THREADS / 32) + (threadIdx.x >> 5);
  const int nw = gridDim.x * (FILTERED_THREADS / 32);
  Counters cnt;
  if (SR != SS_REAL && many_hits) pull_groups<SR, C>(d, k, gbm, sg, wid, nw, cnt);
  else pull_items<SR, C, SS_FORMAT_SLIMSELL, false, true>(d, k, false, gbm, sg, wid, nw, cnt);
  finish_iteration_block<FILTERED_THREADS>(d, cnt.nw, cnt.deg, cnt.slots, cnt.act, cnt.maxdeg,
                                           IterLaunch{variant, cond, use_cond});
}

// Start of a run, thread t0 of `stride`: nothing visited but the root row (none if
// negative), empty frontiers.  The claim words of the rows without neighbours (past
// n_live) are left alone: no pass reads them.
__device__ __forceinline__ void init_rows(const Dev& d, long long t0, long long stride, int root_row,
                                          unsigned long long root_word) {
  ulonglong2* claim2 = reinterpret_cast<ulonglong2*>(d.claim);  // (n_pad is a multiple of 8)
  const long long pairs = (d.n_live + 1) / 2;
  for (long long i = t0; i < pairs; i += stride)
    claim2[i] = make_ulonglong2(2 * i == root_row ? root_word : 0ull, 2 * i + 1 == root_row ? root_word : 0ull);
  if (t0 == 0 && root_row >= 2 * pairs) d.claim[root_row] = root_word;
  for (long long w = t0; w < d.fb_words; w += stride) {
    const unsigned rb = root_row >= 0 && (root_row >> 5) == w ? 1u << (root_row & 31) : 0u;
    d.fb[0][w] = rb;
    d.fb[1][w] = 0u;
    const long long real = d.n - 32 * w;  // rows of this word that are no padding
    d.vis[w] = (real >= 32 ? 0u : real <= 0 ? ~0u : ~0u << real) | rb;
  }
  for (long long s = t0; s < (long long)d.n_split * d.C; s += stride) {
    d.xacc[s] = 0.0f;
    d.xpar[s] = -1;
  }
  if (d.ctl->error | d.ctl->psum_dirty) {  // a previous run left sums behind (or stopped early)
    for (long long r = t0; r < d.n_pad; r += stride) d.psum[r] = 0.0f;
  }
}

// A whole run (init, every level, outputs) on a small graph in one launch, by one
// thread-block cluster.  A small graph's pass is a few microseconds of work behind
// a launch, a control-block read, a grid-wide tail and the next launch, 10 us a level
// (Kronecker 10: 80 us for five levels); here a level costs the pass, a block
// reduction and one hardware cluster barrier.  The barrier orders the level's
// bitmap, visited and value writes before the next level reads them (past L1), and
// the counters travel through distributed shared memory, double-buffered by level
// parity, so every thread takes the same exit.  Rank 0 keeps the control block in
// shared memory and writes it back at the end.  Kronecker 10: 39 us; 64 graphs of scale
// 10 .. 17 in one batch 0.35 ms, 1.65 with a conditional loop of launches each.
template <int SR, int C>
__global__ void __launch_bounds__(PULL_THREADS, 1) k_small(Dev d, SmallIo io, int policy) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int G = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // (a small graph's counters fit 32 bits)
  __shared__ unsigned part[2][SS_LOCAL_CLUSTER_MAX][5];  // every CTA's counters, by level parity
  __shared__ unsigned wpart[PULL_THREADS / 32][5];
  __shared__ Ctl ctl;  // (rank 0)
  const int nw = G * (PULL_THREADS / 32);
  ItemCache* cache = d.n_items <= 32 * nw
                         ? reinterpret_cast<ItemCache*>(ss_smem_bits + SMEM_GUARD + d.smem_words) : nullptr;
  const int root = io.roots ? io.roots[io.i] : io.root;
  const int root_row = d.invperm[root];
  {
    const long long t0 = (long long)rank * PULL_THREADS + tid, stride = (long long)G * PULL_THREADS;
    init_rows(d, t0, stride, root_row, claim_word(0, root));
    if (rank == 0 && tid == PULL_THREADS - 1) {
      d.fr[root_row] = 1.0f;
      init_ctl(d, &ctl, root_row);
    }
  }
  cl.sync();
  unsigned long long reached = 1;
  for (int k = 1;; ++k) {
    const unsigned* gbm = d.fb[(k - 1) & 1];
    Staged sg;
    sg.sm = ss_smem_bits + SMEM_GUARD;
    sg.smf = nullptr;
    sg.sf = 0;
    sg.sbits = d.smem_words * 32;  // the whole bitmap
    if (tid < SMEM_GUARD) ss_smem_bits[tid] = 0u;
    stage_words(gbm, d.smem_words);
    stage_wait();
    Counters cnt;
    pull_items<SR, C, SS_FORMAT_SLIMSELL, true>(d, k, policy == SS_V_FULL, gbm, sg,
                                                rank * (PULL_THREADS / 32) + warp, nw, cnt, cache, k == 1);
    const unsigned v[5] = {(unsigned)cnt.nw, (unsigned)cnt.deg, (unsigned)cnt.slots, (unsigned)cnt.act, cnt.maxdeg};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const unsigned w = i < 4 ? __reduce_add_sync(SS_FULL_MASK, v[i]) : __reduce_max_sync(SS_FULL_MASK, v[i]);
      if (lane == 0) wpart[warp][i] = w;
    }
    __syncthreads();
    if (warp < 5) {  // counter `warp` over the block's warps, told to every CTA
      const unsigned x = lane < PULL_THREADS / 32 ? wpart[lane][warp] : 0u;
      const unsigned w = warp < 4 ? __reduce_add_sync(SS_FULL_MASK, x) : __reduce_max_sync(SS_FULL_MASK, x);
      if (lane < G) cl.map_shared_rank(&part[0][0][0], lane)[((k & 1) * SS_LOCAL_CLUSTER_MAX + rank) * 5 + warp] = w;
    }
    // level k is complete (one CTA alone needs no cluster-wide release of its writes)
    if (G > 1) cl.sync();
    else __syncthreads();
    unsigned tot[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const unsigned x = lane < G ? part[k & 1][lane][i] : 0u;
      tot[i] = i < 4 ? __reduce_add_sync(SS_FULL_MASK, x) : __reduce_max_sync(SS_FULL_MASK, x);
    }
    reached += tot[0];
    if (rank == 0 && tid == PULL_THREADS - 1) advance_level(d, &ctl, k, tot[0], tot[1], tot[2], tot[3], tot[4], policy);
    // the same decision advance_level takes
    if (tot[0] == 0 || k >= d.n + 1 || reached > d.reach_cap) break;
  }
  if (rank == 0) {
    __syncthreads();
    const unsigned* src = reinterpret_cast<const unsigned*>(&ctl);
    unsigned* dst = reinterpret_cast<unsigned*>(d.ctl);
    for (int i = tid; i < (int)(sizeof(Ctl) / sizeof(unsigned)); i += PULL_THREADS) dst[i] = src[i];
  }
  int* dist = io.dists ? io.dists[io.i] : io.dist;
  int* parent = io.parents ? io.parents[io.i] : io.parent;
  if (dist || parent)
    write_outputs(d, dist, parent, root_row, (long long)rank * PULL_THREADS + tid, (long long)G * PULL_THREADS);
}

__global__ void k_init(Dev d) {
  init_rows(d, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, -1, 0ull);
}

__global__ void k_init_root(Dev d, int root) { init_root_state(d, root); }

// DP transformation as a separate pass (Section II-C): the parent of a row at
// level L >= 1 is its largest-id neighbour at level L-1.  Neighbours are stored
// in descending original id, so each lane's first hit in its column sequence is
// that lane's maximum; lanes stop once their rows are resolved.
template <int C>
__global__ void __launch_bounds__(PULL_THREADS, 1) k_dp(Dev d) {
  constexpr int Q = C / 4;
  constexpr int PULL_STEP = SS_PULL_STEP;
  const int lane = threadIdx.x & 31;
  const int wid = blockIdx.x * (PULL_THREADS / 32) + (threadIdx.x >> 5);
  const int nw = gridDim.x * (PULL_THREADS / 32);
  unsigned long long my_slots = 0;
  for (long long b0 = wid; b0 < d.n_items; b0 += 32LL * nw) {
    const long long my_it = b0 + (long long)lane * nw;
    int4 my_item = make_int4(0, 0, 0, -1);
    long long my_start = 0;
    if (my_it < d.n_items) {
      my_item = d.items[my_it];
      my_start = d.cs[my_item.x] + (long long)my_item.y * C;
    }
    unsigned todo = __ballot_sync(SS_FULL_MASK, my_it < d.n_items);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int4 item = shfl_int4(my_item, src);
      const long long start = __shfl_sync(SS_FULL_MASK, my_start, src);
      const int chunk = item.x;
      const int R0 = chunk * C + 4 * (lane % Q);
      // upper halves of the claim words: 0x7fffffff - level, 0 while unvisited;
      // a row's parents are the neighbours whose half is one larger than its own
      int tgt[4];
      int hit[4];
      bool need = false;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int up = (int)(d.claim[R0 + r] >> 32);
        tgt[r] = (up > 0 && up < 0x7fffffff && R0 + r < d.n_live) ? up + 1 : -2;
        hit[r] = -1;
        need |= tgt[r] >= 0;
      }
      const int nq = (item.z - item.y) * Q;
      const int4* base = reinterpret_cast<const int4*>(d.col + start);
      for (int q0 = 0; q0 < nq && __any_sync(SS_FULL_MASK, need); q0 += 32 * PULL_STEP) {
        if (!need) continue;
        int4 c[PULL_STEP];
#pragma unroll
        for (int u = 0; u < PULL_STEP; ++u) {
          const int q = q0 + lane + 32 * u;
          c[u] = (q < nq) ? ld_stream(base + q) : make_int4(-1, -1, -1, -1);
          if (q < nq) my_slots += 4;
        }
        int Lv[PULL_STEP][4];
#pragma unroll
        for (int u = 0; u < PULL_STEP; ++u) {
          Lv[u][0] = (int)(d.claim[max(c[u].x, 0)] >> 32);
          Lv[u][1] = (int)(d.claim[max(c[u].y, 0)] >> 32);
          Lv[u][2] = (int)(d.claim[max(c[u].z, 0)] >> 32);
          Lv[u][3] = (int)(d.claim[max(c[u].w, 0)] >> 32);
        }
        need = false;
#pragma unroll
        for (int u = 0; u < PULL_STEP; ++u) {
          const int cc[4] = {c[u].x, c[u].y, c[u].z, c[u].w};
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (hit[r] < 0 && tgt[r] >= 0 && cc[r] >= 0 && Lv[u][r] == tgt[r]) hit[r] = cc[r];
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) need |= (tgt[r] >= 0 && hit[r] < 0);
      }
      int best[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) best[r] = hit[r] >= 0 ? d.perm[hit[r]] : -1;
#pragma unroll
      for (int off = Q; off < 32; off <<= 1)
#pragma unroll
        for (int r = 0; r < 4; ++r) best[r] = max(best[r], __shfl_xor_sync(SS_FULL_MASK, best[r], off));
      if (lane < Q) {
        if (item.w < 0) {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (tgt[r] >= 0) parent_half(d, R0 + r)[0] = best[r] + 1;
        } else {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (best[r] >= 0) atomicMax(parent_half(d, R0 + r), best[r] + 1);
        }
      }
    }
  }
  __shared__ unsigned long long red[PULL_THREADS / 32];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) my_slots += __shfl_down_sync(SS_FULL_MASK, my_slots, off);
  if (lane == 0) red[threadIdx.x >> 5] = my_slots;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long s = 0;
    for (int w = 0; w < PULL_THREADS / 32; ++w) s += red[w];
    if (s) atomicAdd(&d.ctl->dp_slots, s);
  }
}

// Rows of split chunks start the DP pass at "no parent" (they combine by atomicMax).
__global__ void k_dp_clear(Dev d) {
  for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < d.n_items;
       it += (long long)gridDim.x * blockDim.x) {
    const int4 item = d.items[it];
    if (item.w >= 0 && item.y == 0)
      for (int l = 0; l < d.C; ++l)
        if (item.x * d.C + l < d.n_live && (d.claim[item.x * d.C + l] >> 32) - 1u < 0x7ffffffeu)
          *parent_half(d, item.x * d.C + l) = 0;
  }
}

__global__ void k_output(Dev d, int* dist, int* parent) {
  write_outputs(d, dist, parent, d.ctl->root_row, (long long)blockIdx.x * blockDim.x + threadIdx.x,
                (long long)gridDim.x * blockDim.x);
}

// Real-semiring values f of the last run in original vertex order; rows the run
// did not reach hold stale values and read as 0.
__global__ void k_values(Dev d, float* out) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < d.n;
       v += (long long)gridDim.x * blockDim.x) {
    const int r = d.invperm[v];
    out[v] = final_claim(d, r, d.ctl->root_row) ? d.fr[r] : 0.0f;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// One 1024-thread block per SM, fewer for small work lists (about 128 items
// per block), so that several small graphs can share the GPU.
int pull_grid(const slimsell_graph* h) {
  const long long want = ((long long)h->n_items + 127) / 128;
  return (int)std::max(1LL, std::min((long long)h->num_sms, want));
}

int vertex_grid(const slimsell_graph* h, int threads) {
  const long long want = ((long long)h->n_pad + threads - 1) / threads;
  return (int)std::max(1LL, std::min((long long)8 * h->num_sms, want));
}

template <int SR, int C, int MODE, int FMT>
static ss_status launch_pull(const slimsell_graph* h, const Dev& d, const IterLaunch& il,
                             cudaStream_t st) {
  static std::atomic<unsigned long long> configured{0};
  if (first_on_device(configured))
    SS_CUDA(cudaFuncSetAttribute(k_pull<SR, C, MODE, FMT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SS_SMEM_LIMIT_BYTES));
  k_pull<SR, C, MODE, FMT><<<pull_grid(h), PULL_THREADS, (size_t)(d.smem_words + SMEM_GUARD) * 4, st>>>(
      d, il.variant, il.cond, il.use_cond);
  SS_CUDA(cudaGetLastError());
  return SS_OK;
}

template <int SR, int C>
static ss_status launch_filtered(const slimsell_graph* h, const Dev& d, const IterLaunch& il,
                                 cudaStream_t st) {
  static std::atomic<unsigned long long> configured{0};
  if (first_on_device(configured))
    SS_CUDA(cudaFuncSetAttribute(k_pull_filtered<SR, C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SS_SMEM_LIMIT_BYTES));
  // A level here is a chain of latencies in each warp, so a graph that does not fill the GPU gets
  // a block per FILTERED_ITEMS items, about one a warp.  With pull_grid's 128 (6.4 a warp):
  // a 380 x 380 lattice 6.43 ms, 5.57 so; Kronecker 17 412 us, 211.
  constexpr long long FILTERED_ITEMS = 24;
  const int grid = (int)std::max(1LL, std::min((long long)h->num_sms, (h->n_items + FILTERED_ITEMS - 1) / FILTERED_ITEMS));
  k_pull_filtered<SR, C><<<grid, FILTERED_THREADS, (size_t)(d.smem_words + SMEM_GUARD) * 4, st>>>(
      d, il.variant, il.cond, il.use_cond);
  SS_CUDA(cudaGetLastError());
  return SS_OK;
}

// Graphs whose whole run goes into one launch (k_small): the fixed full and SlimWork
// policies over SlimSell with the whole bitmap staged.  Where a run has the GPU to itself
// that is a graph of up to SMALL_ROWS live rows (8 a thread of one CTA) and SMALL_DENSE_SLOTS
// slots (what 16 CTAs stream in a few microseconds) without items of more than SMALL_ITEM
// slots, one of which would keep a warp busy for longer than the levels' launches take; and any
// graph of up to SMALL_SLOTS slots.  One launch / grid-wide, SlimWork tropical, us a call
// that is waited for:
//   Kronecker 10 in chunks of 32 69 / 118, of 64 93 / 131, of 32 sorted in windows of 256 69 / 118;
//   Kronecker 13 129 / 195, in chunks of 8 91 / 161; G(8 K, 8n) 82 / 165, G(8 K, 60n) 105 / 250;
//   lattice 64^2 422 / 1202; Kronecker 13 in chunks of 64 with items of 16 K slots 193 / 244, of
//   64 K 402 / 388, of 150 K 742 / 616; Kronecker 10 there with one of 30 K 132 / 162, but sel-max
//   over full passes 270 / 256, real 425 / 383, with items of 16 K 170 / 190 and 266 / 278.
// It goes on to gain past SMALL_ROWS (lattice 128^2 823 / 1678, Kronecker 14 154 / 229), but the
// adaptive policies do not run here, and from there on they, who scale, would lose to
// plain SlimWork on small long-diameter graphs.
// In a batch, where graphs run side by side: up to SMALL_BATCH_SLOTS (batch_small); a
// cluster's SMs are a graph's share of the GPU and its size follows from its share of the
// slots (at least SMALL_BATCH_MIN slots a CTA: 32 graphs of scale 10 .. 13 take 171 us,
// 217 with 16 K).
#ifndef SS_SMALL_SLOTS
#define SS_SMALL_SLOTS (32 << 10)
#endif
#ifndef SS_SMALL_SLOTS_PER_CTA
#define SS_SMALL_SLOTS_PER_CTA (16 << 10)
#endif
#ifndef SS_SMALL_BATCH_SLOTS
#define SS_SMALL_BATCH_SLOTS (4 << 20)
#endif
#ifndef SS_SMALL_BATCH_MIN
#define SS_SMALL_BATCH_MIN (64 << 10)
#endif
constexpr long long SMALL_SLOTS = SS_SMALL_SLOTS;                  // one run alone on the GPU
constexpr int SMALL_ROWS = 8 << 10;
constexpr long long SMALL_DENSE_SLOTS = 512 << 10;
constexpr long long SMALL_ITEM = 16 << 10;
constexpr long long SMALL_SLOTS_PER_CTA = SS_SMALL_SLOTS_PER_CTA;
constexpr long long SMALL_BATCH_SLOTS = SS_SMALL_BATCH_SLOTS;      // many side by side
constexpr long long SMALL_BATCH_MIN = SS_SMALL_BATCH_MIN;
constexpr long long SMALL_BATCH_ALONE = 512 << 10;  // slots, or live rows, up to which a graph of a
constexpr int SMALL_BATCH_ROWS = 64 << 10;          // batch is a cluster whatever its company (batch_small)

static bool whole_run(const slimsell_graph* h, const Dev& d, int policy, long long max_slots) {
  return (policy == SS_V_FULL || policy == SS_V_SLIMWORK) && d.format == SS_FORMAT_SLIMSELL &&
         h->slots <= max_slots && (long long)d.smem_words * 32 >= h->n_pad &&
         (long long)d.smem_words * 4 <= SS_SMEM_LIMIT_BYTES - 16 - (long long)sizeof(ItemCache) * PULL_THREADS;
}
static long long longest_item(const slimsell_graph* h) {  // slots
  return (long long)h->C * (h->split_w > 0 ? std::min(h->split_w, h->max_degree) : h->max_degree);
}
static bool run_small(const slimsell_graph* h, const Dev& d, int policy) {
  const bool rows = h->n_live <= SMALL_ROWS && longest_item(h) <= SMALL_ITEM;
  return whole_run(h, d, policy, rows ? SMALL_DENSE_SLOTS : SMALL_SLOTS);
}
static size_t small_smem(const Dev& d) {
  return (size_t)(d.smem_words + SMEM_GUARD) * 4 + sizeof(ItemCache) * PULL_THREADS;
}

// CTAs of the run's cluster: a power of two, at most what the device places.
static int small_cluster(const slimsell_graph* h, long long slots_per_cta) {
  int G = 1;
  while (G < h->local_cluster && G * slots_per_cta < h->slots) G *= 2;
  return G;
}

// CTAs of a graph's cluster in a batch of batch_slots slots, 0 where it cannot run as one.
static int batch_cluster(const slimsell_graph* h, long long batch_slots) {
  return std::min(8, small_cluster(h, std::max(SMALL_BATCH_MIN, batch_slots / h->num_sms)));
}
int batch_ctas(const slimsell_graph* h, const Dev& d, int policy, long long batch_slots) {
  if (h->slots < SMALL_BATCH_MIN) return 0;
  return whole_run(h, d, policy, SMALL_BATCH_SLOTS) ? batch_cluster(h, batch_slots) : 1;
}

// Whether a graph of a batch runs as one cluster or as a loop of grid-wide launches.  A loop's
// passes have the whole GPU, eight CTAs a twentieth of it; but a loop pays its launches, which
// those of other loops queue behind (about 4 us a level and loop), and its grids wait for SMs
// that clusters hold.  So the larger graphs run as clusters only where the batch's clusters,
// those of graphs that earn a CTA or more (ctas), fill the GPU, or two fifths of it where loops
// are slow themselves: for sparse graphs, whose runs are many short levels, and for items past
// SMALL_ITEM, whose one warp the rest of the GPU waits for (four fifths past eight times that,
// which clusters are slow at too).  SlimWork, clusters / loops:
//   Kronecker 16 (2.1 M slots) alone 202 us / 229, 17 (4.1 M) 261 / 192, 16 of 17 536 / 467, 64 1091 / 1648;
//   G(60 K, 8n) (1 M) 175 / 181, G(120 K) (1.9 M) 271 / 188, 16 of it 535 / 476, 64 1056 / 1733;
//   G(200 K) (3.2 M) 434 / 189, 16 of it 868 / 637, 64 1763 / 2363;
//   lattice 300^2 (0.3 M) 2.3 ms / 3.6, 500^2 (0.9 M) 8.7 / 7.8, 16 of it 17.7 / 32.9,
//   900^2 (3.1 M) 56 / 20, 4 of it 62 / 46, 16 of it 113 / 177;
//   64 graphs of Kronecker 10 .. 17 (192 CTAs), all clusters 432 us, those of 17 in loops 503;
//   in chunks of 64 with items of 64 K slots, Kronecker 12 alone 287 / 281, 16 of it 422 / 731,
//   of 260 K, 8 of Kronecker 15 1521 / 1280;
//   finely split (items of 1 K slots) Kronecker 16 alone 200 / 168: past 1 M slots only graphs of
//   longer items are clusters in any company.
bool batch_small(const slimsell_graph* h, const Dev& d, int policy, long long ctas) {
  if (!whole_run(h, d, policy, SMALL_BATCH_SLOTS)) return false;
  if (h->slots <= SMALL_BATCH_MIN) return true;
  const long long item = longest_item(h);
  if (item <= SMALL_ITEM && (h->slots <= SMALL_BATCH_ALONE ||
                             (h->n_live <= SMALL_BATCH_ROWS && (h->slots <= 2 * SMALL_BATCH_ALONE || item >= SMALL_ITEM / 4))))
    return true;
  const int fifths = item > 8 * SMALL_ITEM ? 4 : item > SMALL_ITEM || h->nnz < 8LL * h->n_live ? 2 : 5;
  return ctas >= (long long)fifths * h->num_sms / 5;
}

using SmallKernel = void (*)(Dev, SmallIo, int);

template <int SR>
static SmallKernel small_kernel_c(int C) {
  switch (C) {
    case 8: return k_small<SR, 8>;
    case 16: return k_small<SR, 16>;
    case 32: return k_small<SR, 32>;
    default: return k_small<SR, 64>;
  }
}

// The kernel of a semiring and chunk height, with its launch limits raised.
static ss_status small_kernel(const slimsell_graph* h, int sr, SmallKernel* out) {
  static std::atomic<unsigned long long> configured[4][4];
  const int c = h->C == 8 ? 0 : h->C == 16 ? 1 : h->C == 32 ? 2 : 3;
  *out = sr == SS_TROPICAL ? small_kernel_c<SS_TROPICAL>(h->C)
       : sr == SS_REAL     ? small_kernel_c<SS_REAL>(h->C)
       : sr == SS_BOOLEAN  ? small_kernel_c<SS_BOOLEAN>(h->C)
                           : small_kernel_c<SS_SELMAX>(h->C);
  if (first_on_device(configured[sr][c])) {
    SS_CUDA(cudaFuncSetAttribute(*out, cudaFuncAttributeMaxDynamicSharedMemorySize, SS_SMEM_LIMIT_BYTES));
    SS_CUDA(cudaFuncSetAttribute(*out, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  }
  return SS_OK;
}

static ss_status launch_small(const slimsell_graph* h, const Dev& d, int sr, int policy, const SmallIo& io, int G,
                              cudaStream_t st) {
  SmallKernel kern = nullptr;
  ss_status s = small_kernel(h, sr, &kern);
  if (s != SS_OK) return s;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(PULL_THREADS);
  cfg.dynamicSmemBytes = small_smem(d);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = G;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  SS_CUDA(cudaLaunchKernelEx(&cfg, kern, d, io, policy));
  return SS_OK;
}

ss_status add_small_node(const slimsell_graph* h, const Dev& d, int sr, int policy, const SmallIo& io,
                         long long batch_slots, cudaGraph_t g, cudaGraphNode_t* out) {
  SmallKernel kern = nullptr;
  ss_status s = small_kernel(h, sr, &kern);
  if (s != SS_OK) return s;
  const int G = batch_cluster(h, batch_slots);
  Dev dd = d;
  SmallIo ii = io;
  int pol = policy;
  void* args[] = {&dd, &ii, &pol};
  cudaKernelNodeParams kp = {};
  kp.func = (void*)kern;
  kp.gridDim = dim3(G);
  kp.blockDim = dim3(PULL_THREADS);
  kp.sharedMemBytes = (unsigned)small_smem(d);
  kp.kernelParams = args;
  SS_CUDA(cudaGraphAddKernelNode(out, g, nullptr, 0, &kp));
  cudaKernelNodeAttrValue v = {};
  v.clusterDim.x = G;
  v.clusterDim.y = 1;
  v.clusterDim.z = 1;
  SS_CUDA(cudaGraphKernelNodeSetAttribute(*out, cudaLaunchAttributeClusterDimension, &v));
  return SS_OK;
}

template <int SR, int MODE, int FMT>
static ss_status launch_pull_c(const slimsell_graph* h, const Dev& d, const IterLaunch& il,
                               cudaStream_t st) {
  switch (h->C) {
    case 8: return launch_pull<SR, 8, MODE, FMT>(h, d, il, st);
    case 16: return launch_pull<SR, 16, MODE, FMT>(h, d, il, st);
    case 32: return launch_pull<SR, 32, MODE, FMT>(h, d, il, st);
    default: return launch_pull<SR, 64, MODE, FMT>(h, d, il, st);
  }
}

// The Sell-C-sigma format is instantiated for the full and SlimWork passes only
// (slimsell_bfs accepts it with those policies).
template <int SR>
static ss_status launch_pull_m(const slimsell_graph* h, const Dev& d, int mode, const IterLaunch& il,
                               cudaStream_t st) {
  const bool sell = d.format == SS_FORMAT_SELL;
  switch (mode) {
    case MODE_FULL:
      return sell ? launch_pull_c<SR, MODE_FULL, SS_FORMAT_SELL>(h, d, il, st)
                  : launch_pull_c<SR, MODE_FULL, SS_FORMAT_SLIMSELL>(h, d, il, st);
    case MODE_SLIMWORK:
      return sell ? launch_pull_c<SR, MODE_SLIMWORK, SS_FORMAT_SELL>(h, d, il, st)
                  : launch_pull_c<SR, MODE_SLIMWORK, SS_FORMAT_SLIMSELL>(h, d, il, st);
    default:
      switch (h->C) {
        case 8: return launch_filtered<SR, 8>(h, d, il, st);
        case 16: return launch_filtered<SR, 16>(h, d, il, st);
        case 32: return launch_filtered<SR, 32>(h, d, il, st);
        default: return launch_filtered<SR, 64>(h, d, il, st);
      }
  }
}

static ss_status launch_iteration(const slimsell_graph* h, const Dev& d, int sr, int mode,
                                  const IterLaunch& il, cudaStream_t st) {
  switch (sr) {
    case SS_TROPICAL: return launch_pull_m<SS_TROPICAL>(h, d, mode, il, st);
    case SS_REAL: return launch_pull_m<SS_REAL>(h, d, mode, il, st);
    case SS_BOOLEAN: return launch_pull_m<SS_BOOLEAN>(h, d, mode, il, st);
    default: return launch_pull_m<SS_SELMAX>(h, d, mode, il, st);
  }
}

// Queue the kernels of one iteration of the given variant.  The cluster push
// runs as many small levels as it can per launch (under profiling it times each
// level on the device).
static ss_status launch_variant(const slimsell_graph* h, const Dev& d, int sr, int variant,
                                const IterLaunch& il, cudaStream_t st) {
  switch (variant) {
    case VAR_FULL: return launch_iteration(h, d, sr, MODE_FULL, il, st);
    case VAR_SLIMWORK: return launch_iteration(h, d, sr, MODE_SLIMWORK, il, st);
    case VAR_PUSH: return launch_push(h, d, sr, il, st);
    case VAR_PUSH_LOCAL:
      return launch_push_local(h, d, sr, il, 1 << 30, st);
    default: return launch_iteration(h, d, sr, MODE_FILTERED, il, st);
  }
}

// Policies that choose the variant on the device before every iteration.
static bool adaptive(int policy) {
  return policy == SS_V_PUSH || policy == SS_V_HEURISTIC || policy == SS_V_LEARNED;
}

// Capture the kernels of one variant into graph g (a conditional body).
#ifndef SS_LOOP_UNROLL
#define SS_LOOP_UNROLL 3
#endif

static ss_status capture_into(slimsell_graph* h, const Dev& d, int sr, int variant,
                              const IterLaunch& il, cudaGraph_t g, int reps = 1) {
  cudaStream_t cs = nullptr;
  cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  if (e == cudaSuccess)
    e = cudaStreamBeginCaptureToGraph(cs, g, nullptr, nullptr, 0, cudaStreamCaptureModeRelaxed);
  if (e != cudaSuccess) {
    if (cs) cudaStreamDestroy(cs);
    return cuda_fail(e, "cudaStreamBeginCaptureToGraph");
  }
  ss_status s = SS_OK;
  for (int i = 0; i < reps && s == SS_OK; ++i) s = launch_variant(h, d, sr, variant, il, cs);
  cudaGraph_t captured = nullptr;
  e = cudaStreamEndCapture(cs, &captured);
  cudaStreamDestroy(cs);
  if (s != SS_OK) return s;
  if (e != cudaSuccess) return cuda_fail(e, "cudaStreamEndCapture");
  return SS_OK;
}

// Add one device-side iteration loop to graph g after the given dependencies:
// a conditional WHILE node whose body is the fixed variant's kernels, or (adaptive
// policies) the decide kernel followed by a conditional SWITCH over the five
// executed variants.  The last block of each iteration's final kernel (or the
// single-block push, when it stops or hands back) sets the WHILE condition.
ss_status add_loop_node(slimsell_graph* h, const Dev& d, int sr, int policy, cudaGraph_t g,
                        const cudaGraphNode_t* deps, size_t ndeps, cudaGraphNode_t* out) {
  cudaGraphConditionalHandle cw;
  cudaGraphNodeParams wp = {};
  cudaError_t e = cudaGraphConditionalHandleCreate(&cw, g, 1, cudaGraphCondAssignDefault);
  if (e == cudaSuccess) {
    wp.type = cudaGraphNodeTypeConditional;
    wp.conditional.handle = cw;
    wp.conditional.type = cudaGraphCondTypeWhile;
    wp.conditional.size = 1;
    e = cudaGraphAddNode(out, g, deps, nullptr, ndeps, &wp);
  }
  if (e != cudaSuccess) return cuda_fail(e, "conditional WHILE node");
  cudaGraph_t body = wp.conditional.phGraph_out[0];
  // a fixed variant's body holds SS_LOOP_UNROLL iterations: one more than the
  // run needs returns at once (every kernel checks the done flag first) and
  // leaves the WHILE condition as the finishing iteration set it; three per body
  // measured 2.3 % faster per Kronecker 22 BFS than one (fewer conditional trips)
  if (!adaptive(policy)) return capture_into(h, d, sr, policy, IterLaunch{policy, cw, 1}, body, SS_LOOP_UNROLL);
  cudaGraphConditionalHandle csw;
  cudaGraphNode_t dnode, snode;
  cudaGraphNodeParams sp = {};
  e = cudaGraphConditionalHandleCreate(&csw, body, 0, 0);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGraphConditionalHandleCreate(switch)");
  ss_status s = add_decide_node(h, d, sr, policy, csw, cw, body, &dnode);
  if (s != SS_OK) return s;
  sp.type = cudaGraphNodeTypeConditional;
  sp.conditional.handle = csw;
  sp.conditional.type = cudaGraphCondTypeSwitch;
  sp.conditional.size = N_VARIANTS;
  e = cudaGraphAddNode(&snode, body, &dnode, nullptr, 1, &sp);
  if (e != cudaSuccess) return cuda_fail(e, "conditional SWITCH node");
  for (int v = 0; v < N_VARIANTS && s == SS_OK; ++v)
    s = capture_into(h, d, sr, v, IterLaunch{v, cw, 1}, sp.conditional.phGraph_out[v]);
  return s;
}

void drop_loop_graphs(slimsell_graph* h) {
  for (auto& row : h->loop_exec)
    for (auto& e : row)
      if (e) {
        cudaGraphExecDestroy(e);
        e = nullptr;
      }
}

// The single-call loop graph, built once per (semiring, policy, staged-prefix
// size) and cached in the handle.
static ss_status loop_graph(slimsell_graph* h, const Dev& d, int sr, int policy,
                            cudaGraphExec_t* out) {
  cudaGraphExec_t& slot = h->loop_exec[sr][policy];
  if (slot && h->loop_smem_words[sr][policy] == d.smem_words) {
    *out = slot;
    return SS_OK;
  }
  if (slot) {
    SS_CUDA(cudaGraphExecDestroy(slot));
    slot = nullptr;
  }
  cudaGraph_t g = nullptr;
  SS_CUDA(cudaGraphCreate(&g, 0));
  cudaGraphNode_t wnode;
  ss_status s = add_loop_node(h, d, sr, policy, g, nullptr, 0, &wnode);
  if (s == SS_OK) {
    cudaError_t e = cudaGraphInstantiate(&slot, g, 0);
    if (e != cudaSuccess) {
      slot = nullptr;
      s = cuda_fail(e, "cudaGraphInstantiate");
    }
  }
  cudaGraphDestroy(g);
  if (s != SS_OK) return s;
  h->loop_smem_words[sr][policy] = d.smem_words;
  *out = slot;
  return SS_OK;
}

template <int C>
static ss_status launch_dp_c(const slimsell_graph* h, const Dev& d, cudaStream_t st) {
  k_dp<C><<<h->num_sms, PULL_THREADS, 0, st>>>(d);
  SS_CUDA(cudaGetLastError());
  return SS_OK;
}

static ss_status launch_dp(const slimsell_graph* h, const Dev& d, cudaStream_t st) {
  k_dp_clear<<<4 * h->num_sms, 256, 0, st>>>(d);
  SS_CUDA(cudaGetLastError());
  switch (h->C) {
    case 8: return launch_dp_c<8>(h, d, st);
    case 16: return launch_dp_c<16>(h, d, st);
    case 32: return launch_dp_c<32>(h, d, st);
    default: return launch_dp_c<64>(h, d, st);
  }
}

}  // namespace ss

namespace ss {
// Read back the counters of the last call once its work has finished.
static ss_status finish_run(slimsell_graph* h) {
  if (!h->pending) return SS_OK;
  SS_CUDA(cudaEventSynchronize(h->ev_done));
  h->pending = 0;
  const Ctl& c = *h->h_ctl;
  h->last.iterations = c.k - 1;
  h->last.reached = (long long)c.reached;
  h->last.reached_degree = (long long)c.reached_deg;
  h->last.slots = (long long)c.total_slots;
  h->last.dp_slots = (long long)c.dp_slots;
  if (h->profiling) {
    float ms = 0.f;
    SS_CUDA(cudaEventElapsedTime(&ms, h->ev_c, h->ev_d));
    h->last.total_ms = ms;
  }
  if (c.error) {
    set_error("slimsell_bfs: iteration limit reached (device error flags %d)", c.error);
    return SS_ERR_CUDA;
  }
  return SS_OK;
}
}  // namespace ss

extern "C" {

ss_status slimsell_bfs(slimsell_handle h, int32_t root, int32_t semiring, int32_t policy,
                       int32_t* d_dist, int32_t* d_parent, void* stream) {
  using namespace ss;
  set_error("");
  if (!h) {
    set_error("slimsell_bfs: NULL handle");
    return SS_ERR_INVALID;
  }
  if (root < 0 || root >= h->n) {
    set_error("slimsell_bfs: root %d out of range [0, %d)", root, h->n);
    return SS_ERR_INVALID;
  }
  if (semiring < SS_TROPICAL || semiring > SS_SELMAX) {
    set_error("slimsell_bfs: unknown semiring %d", semiring);
    return SS_ERR_INVALID;
  }
  if (policy < SS_V_FULL || policy > SS_V_LEARNED) {
    set_error("slimsell_bfs: unknown policy %d", policy);
    return SS_ERR_INVALID;
  }
  if (h->format == SS_FORMAT_SELL && policy != SS_V_FULL && policy != SS_V_SLIMWORK) {
    set_error("slimsell_bfs: the Sell-C-sigma format runs the FULL and SLIMWORK policies only");
    return SS_ERR_UNSUPPORTED;
  }
  h->values_semiring = -1;  // set again once this run is queued
  cudaStream_t st = (cudaStream_t)stream;
  if (h->format == SS_FORMAT_SELL && !h->sell_col) {
    if (h->pending) SS_CUDA(cudaEventSynchronize(h->ev_done));
    ss_status s = sell_arrays(h, st);
    if (s != SS_OK) return s;
  }
  Dev d = h->dev();
  if (h->format == SS_FORMAT_SELL) {
    d.format = SS_FORMAT_SELL;
    d.scol = h->sell_col;
    d.sval = semiring == SS_TROPICAL ? h->sell_vtrop : h->sell_vmul;
  }
  const int grid = vertex_grid(h, 256);
  const bool prof = h->profiling != 0;
  const bool device_loop = h->device_loop && !prof;
  // the previous call's statistics are dropped without waiting for it: its work is
  // ahead of this call's on the same stream (the handle's contract), and a host
  // wait here left the GPU idle between back-to-back runs
  h->pending = 0;
  h->iter_ns.clear();
  double iter_ms = 0.0;
  if (prof) SS_CUDA(cudaEventRecord(h->ev_c, st));

  const bool dp = d_parent && semiring != SS_SELMAX && h->dp_pass;
  const bool whole = device_loop && run_small(h, d, policy);
  if (!whole) {
    k_init<<<grid, 256, 0, st>>>(d);
    k_init_root<<<1, 1, 0, st>>>(d, root);
    SS_CUDA(cudaGetLastError());
  }

  if (whole) {
    SmallIo io{};
    io.root = root;
    io.dist = dp ? nullptr : d_dist;  // (with the DP pass, the outputs follow it)
    io.parent = dp ? nullptr : d_parent;
    ss_status s = launch_small(h, d, semiring, policy, io, small_cluster(h, SMALL_SLOTS_PER_CTA), st);
    if (s != SS_OK) return s;
  } else if (device_loop) {
    cudaGraphExec_t exec = nullptr;
    ss_status s = loop_graph(h, d, semiring, policy, &exec);
    if (s != SS_OK) return s;
    SS_CUDA(cudaGraphLaunch(exec, st));
  } else if (!adaptive(policy) && h->profile_queue) {
    // fixed variant: iterations are queued QUEUE_BATCH at a time, each launch
    // bracketed by its own event pair when profiling, and the host reads the
    // counter once per batch; launches queued past the end of the run return
    // at once (every kernel checks the done flag) and their times are dropped
    constexpr int QUEUE_BATCH = 8;
    if (prof && h->evq.size() < 2 * (size_t)QUEUE_BATCH) {
      while (h->evq.size() < 2 * (size_t)QUEUE_BATCH) {
        cudaEvent_t e = nullptr;
        SS_CUDA(cudaEventCreate(&e));
        h->evq.push_back(e);
      }
    }
    const long long max_iter = (long long)h->n + 2;
    for (long long it = 0;;) {
      if (it > max_iter) {
        set_error("slimsell_bfs: no convergence after %lld iterations", it);
        return SS_ERR_CUDA;
      }
      for (int j = 0; j < QUEUE_BATCH; ++j) {
        ss_status s = launch_decide(h, d, semiring, policy, 0, 0, st);  // logs the iteration's features
        if (s != SS_OK) return s;
        if (prof) SS_CUDA(cudaEventRecord(h->evq[2 * j], st));
        s = launch_variant(h, d, semiring, policy, IterLaunch{policy, 0, 0}, st);
        if (s != SS_OK) return s;
        if (prof) SS_CUDA(cudaEventRecord(h->evq[2 * j + 1], st));
      }
      SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
      SS_CUDA(cudaStreamSynchronize(st));
      const long long ran = (long long)h->h_ctl->k - 1;  // iterations the run has made so far
      if (prof)
        for (int j = 0; j < QUEUE_BATCH && it + j < ran; ++j) {
          float ms = 0.f;
          SS_CUDA(cudaEventElapsedTime(&ms, h->evq[2 * j], h->evq[2 * j + 1]));
          iter_ms += ms;
          h->iter_ns.push_back((int)(ms * 1.0e6f));
        }
      it += QUEUE_BATCH;
      if (h->h_ctl->done) break;
    }
  } else {
    const long long max_iter = (long long)h->n + 2;
    for (long long it = 0;; ++it) {
      if (it > max_iter) {
        set_error("slimsell_bfs: no convergence after %lld iterations", it);
        return SS_ERR_CUDA;
      }
      // the decide kernel logs the iteration's features; adaptive policies read its choice
      ss_status s = launch_decide(h, d, semiring, policy, 0, 0, st);
      if (s != SS_OK) return s;
      int variant = policy;
      if (adaptive(policy)) {
        SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
        SS_CUDA(cudaStreamSynchronize(st));
        variant = h->h_ctl->variant;
      }
      const int k_before = h->h_ctl->k;  // valid when the cluster push is chosen (adaptive)
      if (prof) SS_CUDA(cudaEventRecord(h->ev_a, st));
      s = launch_variant(h, d, semiring, variant, IterLaunch{variant, 0, 0}, st);
      if (s != SS_OK) return s;
      if (prof) SS_CUDA(cudaEventRecord(h->ev_b, st));
      SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
      SS_CUDA(cudaStreamSynchronize(st));
      if (prof) {
        float ms = 0.f;
        SS_CUDA(cudaEventElapsedTime(&ms, h->ev_a, h->ev_b));
        iter_ms += ms;
        h->iter_ns.push_back((int)(ms * 1.0e6f));
        // levels run inside one cluster-push launch were timed on the device;
        // slimsell_get_run_stats takes them from there (marker -1)
        if (variant == VAR_PUSH_LOCAL)  // (k_before is fresh: adaptive policies read ctl above)
          for (int extra = h->h_ctl->k - k_before - 1; extra > 0; --extra) h->iter_ns.push_back(-1);
      }
      if (h->h_ctl->done) break;
    }
  }

  if (dp) {
    ss_status s = launch_dp(h, d, st);
    if (s != SS_OK) return s;
  }
  if ((!whole || dp) && (d_dist || d_parent)) {
    k_output<<<grid, 256, 0, st>>>(d, d_dist, d_parent);
    SS_CUDA(cudaGetLastError());
  }
  if (prof) SS_CUDA(cudaEventRecord(h->ev_d, st));
  SS_CUDA(cudaMemcpyAsync(h->h_ctl, h->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaEventRecord(h->ev_done, st));
  h->last.semiring = semiring;
  h->values_semiring = semiring;
  h->last.iter_kernel_ms = iter_ms;
  h->last.total_ms = 0.0;
  h->pending = 1;
  if (!device_loop) return finish_run(h);
  return SS_OK;
}

ss_status slimsell_get_values(slimsell_handle h, float* d_out, void* stream) {
  using namespace ss;
  set_error("");
  if (!h || !d_out) {
    set_error("slimsell_get_values: NULL argument");
    return SS_ERR_INVALID;
  }
  if (h->values_semiring != SS_REAL) {
    set_error("slimsell_get_values: the handle's last run was not a real-semiring slimsell_bfs");
    return SS_ERR_INVALID;
  }
  const Dev d = h->dev();
  k_values<<<vertex_grid(h, 256), 256, 0, (cudaStream_t)stream>>>(d, d_out);
  SS_CUDA(cudaGetLastError());
  return SS_OK;
}

ss_status slimsell_get_run_stats(slimsell_handle h, ss_run_stats* out, ss_iter_stats* h_iters,
                                 int32_t cap) {
  if (!h || !out) {
    ss::set_error("slimsell_get_run_stats: NULL argument");
    return SS_ERR_INVALID;
  }
  ss_status s = ss::finish_run(h);
  *out = h->last;
  if (h_iters && cap > 0) {
    int cnt = h->last.iterations + 1;
    if (cnt > cap) cnt = cap;
    if (cnt > h->iter_cap) cnt = h->iter_cap;
    SS_CUDA(cudaMemcpy(h_iters, h->iters, sizeof(ss_iter_stats) * (size_t)cnt, cudaMemcpyDeviceToHost));
    // host events time each launch; a launch that ran several levels (cluster
    // push) left -1 markers for its later levels, whose device-side times are
    // taken from the iteration records and moved out of the launch's first level
    int owner = -1;
    for (int i = 0; i < cnt; ++i) {
      const int host = (i >= 1 && i - 1 < (int)h->iter_ns.size()) ? h->iter_ns[i - 1] : 0;
      if (host >= 0) {
        h_iters[i].kernel_ns = host;
        owner = i;
      } else {
        if (owner >= 1) h_iters[owner].kernel_ns = std::max(0, h_iters[owner].kernel_ns - h_iters[i].kernel_ns);
      }
    }
  }
  return s;
}

ss_status slimsell_set_profiling(slimsell_handle h, int32_t on) {
  if (!h) {
    ss::set_error("slimsell_set_profiling: NULL handle");
    return SS_ERR_INVALID;
  }
  h->profiling = on ? 1 : 0;
  return SS_OK;
}

ss_status slimsell_set_option(slimsell_handle h, int32_t option, int64_t value) {
  if (!h) {
    ss::set_error("slimsell_set_option: NULL handle");
    return SS_ERR_INVALID;
  }
  // options change captured loops and buffers a queued run may still be using
  if (h->pending) SS_CUDA(cudaEventSynchronize(h->ev_done));
  switch (option) {
    case SS_OPT_DP_PASS:
      h->dp_pass = value ? 1 : 0;
      return SS_OK;
    case SS_OPT_DEVICE_LOOP:
      h->device_loop = value ? 1 : 0;
      return SS_OK;
    case SS_OPT_PROFILE_QUEUE:
      h->profile_queue = value ? 1 : 0;
      return SS_OK;
    case SS_OPT_FORMAT:
      if (value != SS_FORMAT_SLIMSELL && value != SS_FORMAT_SELL) {
        ss::set_error("slimsell_set_option: format must be SS_FORMAT_SLIMSELL or SS_FORMAT_SELL");
        return SS_ERR_INVALID;
      }
      h->format = (int)value;
      ss::drop_loop_graphs(h);  // captured loops hold the previous kernels
      return SS_OK;
    case SS_OPT_PUSH_BLOCKS:
      if (value < 0 || value > 2) {
        ss::set_error("slimsell_set_option: push blocks must be 0, 1 or 2");
        return SS_ERR_INVALID;
      }
      h->push_blocks = (int)value;
      ss::drop_loop_graphs(h);  // captured loops hold the previous value
      return SS_OK;
    case SS_OPT_SELECTOR_MARGIN:
      if (value < 0 || value > 100000) {
        ss::set_error("slimsell_set_option: selector margin must be in [0, 100000] thousandths");
        return SS_ERR_INVALID;
      }
      h->sel_margin = (float)value / 1000.0f;
      ss::drop_loop_graphs(h);
      return SS_OK;
    case SS_OPT_SMEM_BYTES:
      if (value < 0 || value > SS_SMEM_MAX_BYTES) {
        ss::set_error("slimsell_set_option: shared-memory bytes must be in [0, %d]", SS_SMEM_MAX_BYTES);
        return SS_ERR_INVALID;
      }
      h->smem_bytes = (int)value;
      return SS_OK;
    default:
      ss::set_error("slimsell_set_option: unknown option %d", option);
      return SS_ERR_INVALID;
  }
}

}  // extern "C"
