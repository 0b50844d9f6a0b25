// Betweenness centrality on the SlimSell layout: Brandes' dependency
// accumulation, one of the algorithms the paper names in its conclusion as a
// target for SlimSell, run for up to 64 sources at once.
//
//   levels    the bit-packed multi-source BFS (the boolean semiring of Section
//             III-A on 64-source words, ss_multi.cu) gives, per level L, the
//             word LF[L][v] whose bit s says that v is at distance L from
//             source s; every level's word is kept;
//   forward,  level L = 1, 2, ...: each row v with LF[L][v] != 0 sums, for
//             every such source s, sigma[u][s] over its neighbours u with bit s
//             in LF[L-1][u] (the real-semiring step with the path counts kept);
//   backward, level L = D-1 .. 1: each row v at level L for source s sums
//             t[w][s] = (1 + delta[w][s]) / sigma[w][s] over its neighbours w
//             at level L+1 for s; then delta[v][s] = sigma[v][s] * sum and
//             bc(v) += delta[v][s].
//
// The rows of a level are cut into units of PUSH_UNIT neighbours (hub rows
// spread over many warps); one warp takes a unit, its lanes own sources
// (lane, lane + 32), and the 32 lanes first load 32 neighbours and their level
// words at once, then walk them together, each lane reading the per-source
// values of its two sources (one coalesced row per neighbour).  The units of one
// row add into sigma / the dependency sums with atomics.
//
// Arithmetic.  GB300 has two fp64 lanes per SM: a warp-wide fp64 add holds the pipe
// for 16 clocks, and two of them per visited neighbour (whatever the mask says)
// were 49 of the 62 ms of a Kronecker 22 batch.  So both sums run on the integer
// pipes, and only the post-processing uses fp64:
//   path counts   64-bit integers (exact; in fp64 they were exact below 2^53).
//                 Before each level the host checks that the largest count so far
//                 times the largest degree stays below 2^63;
//   dependencies  t is 128-bit fixed point with F fraction bits.  The t of a row's
//                 dependents sum to at most n (delta = sigma * sum <= n), so
//                 F = 126 - bits(n), and t >= 1 / sigma keeps 60 significant bits as
//                 long as sigma < 2^(F - 60) (2^43 on Kronecker 22).  Fixed-point
//                 sums are exact, whatever their order.
// Counts past either limit (long lattices) go on in fp64 from that point:
// sums then round in no fixed order.  A (vertex, source) pair has one level, so its
// dependency sum and its t share one 16-byte slot.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "ss_device.cuh"

namespace ss {

namespace {

constexpr int BCM_S = 64;  // sources per batch: one bit-packed word per row

// How the per-source values of a pass are held.
enum { BC_COUNT = 0, BC_FP64 = 1, BC_FIXED = 2 };

struct BcScratch {
  void* sigma = nullptr;    // [n_pad][64] shortest-path counts: uint64, or fp64 past 2^63
  void* dep = nullptr;      // [n_pad][64] x 16 bytes: the dependency sum of a pair's own level, then
                            // its t (fixed point), or fp64 t [n_pad][64] | sums [n_pad][64]
  std::vector<unsigned long long*> lf;  // per level: [n_pad] level words
};

std::mutex g_bc_mu;
std::unordered_map<const slimsell_graph*, BcScratch> g_bc;

// The rows of more than one unit add into their slots, so those start at zero
// (the others are stored whole); one warp per row.
__global__ void __launch_bounds__(256) k_bcm_init(Dev d, unsigned long long* sigma, ulonglong2* dep) {
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long r0 = wid * 32; r0 < d.n_pad; r0 += nw * 32) {
    unsigned long_rows = __ballot_sync(SS_FULL_MASK, r0 + lane < d.n_pad && d.rdeg[r0 + lane] > PUSH_UNIT);
    while (long_rows) {
      const long long r = r0 + __ffs(long_rows) - 1;
      long_rows &= long_rows - 1;
      for (int s = lane; s < BCM_S; s += 32) {
        sigma[r * BCM_S + s] = 0ull;
        dep[r * BCM_S + s] = make_ulonglong2(0ull, 0ull);
      }
    }
  }
}

// sigma = 1 for every source at its own row (level 0).
__global__ void k_bcm_roots(Dev d, const int* roots, int kb, unsigned long long* sigma) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < kb) sigma[(long long)d.invperm[roots[s]] * BCM_S + s] = 1ull;
  if (s == 0) d.ctl->count_bits = 1ull;
}

// Path counts so far into fp64, in place (whole rows of any level word set).
__global__ void k_bcm_to_fp64(Dev d, void* sigma) {
  const long long total = (long long)d.n_pad * BCM_S;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x)
    reinterpret_cast<double*>(sigma)[i] = (double)reinterpret_cast<unsigned long long*>(sigma)[i];
}

// fp64 dependency sums of the rows of more than one unit start at zero.
__global__ void __launch_bounds__(256) k_bcm_zero_fp64(Dev d, double* sums) {
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long r = wid; r < d.n_pad; r += nw)
    if (d.rdeg[r] > PUSH_UNIT)
      for (int s = lane; s < BCM_S; s += 32) sums[r * BCM_S + s] = 0.0;
}

// Word 0 of every row of the multi-source frontier (W words per row) into lf.
__global__ void k_bcm_keep(Dev d, const unsigned long long* F, int W, unsigned long long* lf) {
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < d.n_pad;
       r += (long long)gridDim.x * blockDim.x)
    lf[r] = F[r * W];
}

// Work units of the rows with a non-zero level word.
__global__ void __launch_bounds__(256) k_bcm_expand(Dev d, const unsigned long long* lf) {
  const int lane = threadIdx.x & 31;
  const long long stride = ((long long)gridDim.x * blockDim.x) & ~31LL;
  for (long long r0 = (long long)blockIdx.x * blockDim.x + threadIdx.x - lane; r0 < d.n_pad; r0 += stride) {
    const long long r = r0 + lane;
    emit_units(d, (r < d.n_pad && lf[r] != 0ull) ? (int)r : -1, lane);
  }
}

// The value of one (row, source) pair and its sum, by kind.
template <int KIND>
struct BcVal;
template <>
struct BcVal<BC_COUNT> {
  using T = unsigned long long;
  T v = 0ull;
  static __device__ __forceinline__ T zero() { return 0ull; }
  __device__ __forceinline__ void add(T x) { v += x; }
  __device__ __forceinline__ void store(T* p) const { *p = v; }
  __device__ __forceinline__ unsigned long long merge(T* p) const { return v ? atomicAdd(p, v) + v : 0ull; }
  __device__ __forceinline__ unsigned long long bits() const { return v; }
};
template <>
struct BcVal<BC_FP64> {
  using T = double;
  T v = 0.0;
  static __device__ __forceinline__ T zero() { return 0.0; }
  // (a skipped fp64 add frees the pipe, which an fp64 comparison would hold as long: eight of them
  // to a group of gathers made lattices' levels 1.08 times slower)
  __device__ __forceinline__ void add(T x) {
    if (__double_as_longlong(x) != 0) v += x;
  }
  __device__ __forceinline__ void store(T* p) const { *p = v; }
  __device__ __forceinline__ unsigned long long merge(T* p) const {
    if (__double_as_longlong(v) != 0) atomicAdd(p, v);
    return 0ull;
  }
  __device__ __forceinline__ unsigned long long bits() const { return 0ull; }
};
template <>
struct BcVal<BC_FIXED> {
  using T = ulonglong2;  // x low, y high
  unsigned long long lo = 0ull, hi = 0ull;
  static __device__ __forceinline__ T zero() { return make_ulonglong2(0ull, 0ull); }
  __device__ __forceinline__ void add(T q) {
    lo += q.x;
    hi += q.y + (lo < q.x ? 1ull : 0ull);
  }
  __device__ __forceinline__ void store(T* p) const { *p = make_ulonglong2(lo, hi); }
  // the add whose low half wraps carries into the high half, so the total is exact
  __device__ __forceinline__ unsigned long long merge(T* p) const {
    unsigned long long c = hi;
    if (lo) c += atomicAdd(&p->x, lo) + lo < lo ? 1ull : 0ull;
    if (c) atomicAdd(&p->y, c);
    return 0ull;
  }
  __device__ __forceinline__ unsigned long long bits() const { return 0ull; }
};

// One unit: for every neighbour x of row v (in this unit) and every source s in
// lf_v[v] & lf_x[x], add val[x][s] into out[v][s].  Forward: lf_v = LF[L],
// lf_x = LF[L-1], val = out = sigma.  Backward: lf_v = LF[L], lf_x = LF[L+1],
// val = t, out = the sums.  A row of one unit is stored, others are merged.
// ctl->count_bits collects the bits of every finished path count.
#ifndef SS_BC_GATHER
#define SS_BC_GATHER 4
#endif
constexpr int GATHER = SS_BC_GATHER;
template <int KIND>
__global__ void __launch_bounds__(256) k_bcm_gather(Dev d, const unsigned long long* __restrict__ lf_v,
                                                    const unsigned long long* __restrict__ lf_x,
                                                    const typename BcVal<KIND>::T* val,
                                                    typename BcVal<KIND>::T* out) {
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long nunits = min((long long)d.ctl->units, d.units_cap);
  unsigned long long seen = 0ull;
  for (long long ui = wid; ui < nunits; ui += nw) {
    const int2 un = d.units[ui];
    const long long v = un.x;
    const unsigned long long mv = lf_v[v];
    const int deg = d.rdeg[v];
    const int end = min(deg, un.y + PUSH_UNIT);
    const long long chunk = v / d.C;
    const long long base = d.cs[chunk] + (v - chunk * d.C);
    BcVal<KIND> a0, a1;
    for (int j0 = un.y; j0 < end; j0 += 32) {
      const int j = j0 + lane;
      int x = 0;
      unsigned long long mx = 0ull;
      if (j < end) {
        x = __ldg(d.col + base + (long long)j * d.C);
        mx = __ldg(lf_x + x) & mv;
      }
      unsigned any = __ballot_sync(SS_FULL_MASK, mx != 0ull);
      // the neighbours holding a source of this row, GATHER at a time: every load of the group
      // before the first add, which otherwise waits out a memory latency per neighbour
      // (64 sources on Kronecker 22: 40.6 ms, 36.7 so)
      while (any) {
        typename BcVal<KIND>::T x0[GATHER], x1[GATHER];
#pragma unroll
        for (int t = 0; t < GATHER; ++t) {
          const int q = any ? __ffs(any) - 1 : 0;
          unsigned mlo = __shfl_sync(SS_FULL_MASK, (unsigned)mx, q);
          unsigned mhi = __shfl_sync(SS_FULL_MASK, (unsigned)(mx >> 32), q);
          const typename BcVal<KIND>::T* row = val + (long long)__shfl_sync(SS_FULL_MASK, x, q) * BCM_S + lane;
          if (!any) mlo = mhi = 0u;
          any &= any - 1;
          x0[t] = (mlo >> lane & 1u) ? *row : BcVal<KIND>::zero();
          x1[t] = (mhi >> lane & 1u) ? row[32] : BcVal<KIND>::zero();
        }
#pragma unroll
        for (int t = 0; t < GATHER; ++t) {
          a0.add(x0[t]);
          a1.add(x1[t]);
        }
      }
    }
    typename BcVal<KIND>::T* const o = out + v * BCM_S + lane;
    if (deg <= PUSH_UNIT) {
      if (mv >> lane & 1ull) a0.store(o);
      if (mv >> (lane + 32) & 1ull) a1.store(o + 32);
      seen |= a0.bits() | a1.bits();
    } else {
      seen |= a0.merge(o) | a1.merge(o + 32);  // (a row's last merge sees its whole count)
    }
  }
  if (KIND == BC_COUNT) {
    const unsigned lo = __reduce_or_sync(SS_FULL_MASK, (unsigned)seen);
    const unsigned hi = __reduce_or_sync(SS_FULL_MASK, (unsigned)(seen >> 32));
    if (lane == 0 && (lo | hi)) atomicOr(&d.ctl->count_bits, ((unsigned long long)hi << 32) | lo);
  }
}

// 2^125 / m for m in [2^63, 2^64), within 2^-59 of it relatively: Newton-Raphson
// on the reciprocal (y <- y (2 - m y)) in integers, from a float start: 21, 42 and
// then 60 bits.
__device__ __forceinline__ unsigned long long recip_norm(unsigned long long m) {
  const float f = __frcp_rn(__uint2float_rz((unsigned)(m >> 40)) * 1.1920928955078125e-07f);  // 2^63 / m, (1/2, 1]
  unsigned long long y = (unsigned long long)min((unsigned)(f * 4194304.0f), 4194303u) << 40;  // f x 2^62
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    // m y / 2^64 is 2^61 times (1 + e): y += y * (-e)
    const long long e = (long long)((1ull << 61) - __umul64hi(m, y));
    // y * e / 2^61 = ((y << 1) * (e << 2)) >> 64 (y < 2^62, |e| <= 2^41)
    y += (unsigned long long)__mul64hi((long long)(y << 1), e << 2);
  }
  return y;
}

// A 128-bit fixed-point value (scale = 2^-F) as the nearest double.
__device__ __forceinline__ double fixed_to_double(unsigned long long lo, unsigned long long hi, int F) {
  if (!(hi | lo)) return 0.0;
  const int z = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
  // normalise to bit 127; m = the top 64 bits, the rest only breaks ties
  if (z >= 64) {
    hi = lo;
    lo = 0ull;
  }
  const int b = z & 63;
  unsigned long long m = b ? (hi << b) | (lo >> (64 - b)) : hi;
  const unsigned long long rest = lo << b;
  unsigned long long keep = m >> 11;  // 53 bits
  const unsigned tail = (unsigned)m & 0x7FFu;
  if (tail > 0x400u || (tail == 0x400u && (rest != 0ull || (keep & 1ull)))) ++keep;  // to nearest, ties to even
  // value = keep * 2^(127 - z - 52 - F); the carry of a rounding to 2^53 lands in the exponent
  const int e = 127 - z - F + 1023;
  return __longlong_as_double((long long)(((unsigned long long)(e - 1) << 52) + keep));
}

// Backward post of level L: delta = sigma * sum for the row's sources at level L
// (leaf: the deepest level, whose sums are 0), bc += their sum, and the pair's
// slot becomes t = sum + 1 / sigma.  A warp takes up to 32 rows' level words at once
// (fewer on a small graph, whose rows then spread over the warps: 13 sources on
// Kronecker 10 took 717 us with 32 rows a warp always, and take 595).
__global__ void __launch_bounds__(256) k_bcm_post_fixed(Dev d, const unsigned long long* __restrict__ lf,
                                                        const unsigned long long* __restrict__ sigma,
                                                        ulonglong2* dep, int F, int leaf, double* bc) {
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  const int per = (int)min(32LL, (d.n_pad + nw - 1) / nw);
  for (long long r0 = wid * per; r0 < d.n_pad; r0 += nw * per) {
    const unsigned long long word = lane < per && r0 + lane < d.n_pad ? lf[r0 + lane] : 0ull;
    unsigned rows = __ballot_sync(SS_FULL_MASK, word != 0ull);
    while (rows) {
      const int q = __ffs(rows) - 1;
      rows &= rows - 1;
      const long long v = r0 + q;
      const unsigned long long mv = __shfl_sync(SS_FULL_MASK, word, q);
      double sum = 0.0;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int sidx = lane + 32 * h;
        if (mv >> sidx & 1ull) {
          const long long i = v * BCM_S + sidx;
          const unsigned long long sg = sigma[i];
          unsigned long long lo = 0ull, hi = 0ull;
          if (!leaf) {
            const ulonglong2 q2 = dep[i];
            lo = q2.x;
            hi = q2.y;
            if (lo | hi) sum += (double)sg * fixed_to_double(lo, hi, F);
          }
          // 1 / sigma in fixed point: 2^F / sigma = recip_norm(m) * 2^(F + z - 125), m = sigma * 2^z
          const int z = __clzll((long long)sg);
          unsigned long long add_lo, add_hi;
          if ((sg & (sg - 1)) == 0ull) {  // a power of two: exact
            const int e = F - (63 - z);
            add_hi = e >= 64 ? 1ull << (e - 64) : 0ull;
            add_lo = e >= 64 ? 0ull : 1ull << e;
          } else {
            const unsigned long long y = recip_norm(sg << z);
            const int sh = F + z - 125;
            if (sh >= 0) {
              add_lo = sh < 64 ? y << sh : 0ull;
              add_hi = sh == 0 ? 0ull : sh < 64 ? y >> (64 - sh) : y << (sh - 64);
            } else {
              add_lo = y >> -sh;
              add_hi = 0ull;
            }
          }
          lo += add_lo;
          hi += add_hi + (lo < add_lo ? 1ull : 0ull);
          dep[i] = make_ulonglong2(lo, hi);
        }
      }
      if (leaf) continue;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(SS_FULL_MASK, sum, off);
      if (lane == 0 && sum != 0.0) bc[d.perm[v]] += sum;
    }
  }
}

// The same in fp64, one warp per row: t = (1 + delta) / sigma.
__global__ void __launch_bounds__(256) k_bcm_post_fp64(Dev d, const unsigned long long* __restrict__ lf,
                                                       const double* __restrict__ sigma,
                                                       const double* __restrict__ sums, double* t, int leaf,
                                                       double* bc) {
  const int lane = threadIdx.x & 31;
  const long long wid = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long v = wid; v < d.n_pad; v += nw) {
    const unsigned long long mv = lf[v];
    if (!mv) continue;
    double sum = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int sidx = lane + 32 * h;
      if (mv >> sidx & 1ull) {
        const long long i = v * BCM_S + sidx;
        const double sg = sigma[i];
        const double delta = leaf ? 0.0 : sg * sums[i];
        sum += delta;
        t[i] = (1.0 + delta) / sg;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) sum += __shfl_down_sync(SS_FULL_MASK, sum, off);
    if (lane == 0 && sum != 0.0) bc[d.perm[v]] += sum;
  }
}

// Host rules (see the head of this file); count_bits has every bit of every path
// count so far set, so the largest count is below the next power of two.
int bit_length(unsigned long long x) { return x ? 64 - __builtin_clzll(x) : 0; }
bool bc_counts_fit(unsigned long long count_bits, int max_degree) {
  return bit_length(count_bits) + bit_length((unsigned long long)max_degree) <= 63;
}
int bc_fraction_bits(int n) { return 126 - bit_length((unsigned long long)n); }
bool bc_dependencies_fit(unsigned long long count_bits, int F) { return bit_length(count_bits) <= F - 60; }

ss_status bc_scratch(slimsell_graph* h, BcScratch** out) {
  std::lock_guard<std::mutex> lock(g_bc_mu);
  BcScratch& b = g_bc[h];
  const size_t np = (size_t)h->n_pad * BCM_S;
  ss_status s;  // allocate whatever a failed earlier call left missing
  if (!b.sigma && (s = dmalloc(h, (void**)&b.sigma, sizeof(double) * np)) != SS_OK) return s;
  if (!b.dep && (s = dmalloc(h, (void**)&b.dep, sizeof(ulonglong2) * np)) != SS_OK) return s;
  *out = &b;
  return SS_OK;
}

ss_status bc_level_word(slimsell_graph* h, BcScratch* b, size_t L, unsigned long long** out) {
  std::lock_guard<std::mutex> lock(g_bc_mu);
  while (b->lf.size() <= L) {
    unsigned long long* p = nullptr;
    ss_status s = dmalloc(h, (void**)&p, sizeof(unsigned long long) * (size_t)h->n_pad);
    if (s != SS_OK) return s;
    b->lf.push_back(p);
  }
  *out = b->lf[L];
  return SS_OK;
}

}  // namespace

void bc_release(slimsell_graph* h) {
  std::lock_guard<std::mutex> lock(g_bc_mu);
  auto it = g_bc.find(h);
  if (it == g_bc.end()) return;
  BcScratch& b = it->second;
  void* ptrs[] = {b.sigma, b.dep};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  for (unsigned long long* p : b.lf) cudaFree(p);
  g_bc.erase(it);
}

}  // namespace ss

extern "C" ss_status slimsell_bc(slimsell_handle h, const int32_t* d_sources, int32_t k, double* d_bc,
                                 double* kernel_ms, void* stream) {
  using namespace ss;
  set_error("");
  if (!h || !d_sources || !d_bc) {
    set_error("slimsell_bc: NULL argument");
    return SS_ERR_INVALID;
  }
  h->values_semiring = -1;
  if (k < 1) {
    set_error("slimsell_bc: k must be at least 1 (got %d)", k);
    return SS_ERR_INVALID;
  }
  cudaStream_t st = (cudaStream_t)stream;
  std::vector<int> src((size_t)k);
  SS_CUDA(cudaMemcpyAsync(src.data(), d_sources, sizeof(int) * (size_t)k, cudaMemcpyDeviceToHost, st));
  SS_CUDA(cudaStreamSynchronize(st));
  for (int q = 0; q < k; ++q)
    if (src[(size_t)q] < 0 || src[(size_t)q] >= h->n) {
      set_error("slimsell_bc: source %d of entry %d out of range", src[(size_t)q], q);
      return SS_ERR_INVALID;
    }
  if (h->pending) SS_CUDA(cudaEventSynchronize(h->ev_done));
  h->pending = 0;
  BcScratch* b = nullptr;
  ss_status s = bc_scratch(h, &b);
  if (s != SS_OK) return s;
  SS_CUDA(cudaMemsetAsync(d_bc, 0, sizeof(double) * (size_t)h->n, st));
  const int grid = 8 * h->num_sms;
  double ms_sum = 0.0;
  float ms = 0.f;
  auto tic = [&]() -> ss_status {
    if (kernel_ms) SS_CUDA(cudaEventRecord(h->ev_a, st));
    return SS_OK;
  };
  auto toc = [&]() -> ss_status {
    if (kernel_ms) {
      SS_CUDA(cudaEventRecord(h->ev_b, st));
      SS_CUDA(cudaEventSynchronize(h->ev_b));
      SS_CUDA(cudaEventElapsedTime(&ms, h->ev_a, h->ev_b));
      ms_sum += ms;
    }
    return SS_OK;
  };
  for (int b0 = 0; b0 < k; b0 += BCM_S) {
    const int kb = std::min(BCM_S, k - b0);
    if ((s = tic()) != SS_OK) return s;  // (the timed spans leave out the host's per-level reads)
    MultiDev m;
    int W = 1;
    if ((s = multi_start(h, d_sources + b0, kb, st, &m, &W)) != SS_OK) return s;
    const Dev d = m.d;
    unsigned long long* const count = (unsigned long long*)b->sigma;
    double* const sigma = (double*)b->sigma;
    ulonglong2* const dep = (ulonglong2*)b->dep;
    double* const t64 = (double*)b->dep;
    double* const sum64 = t64 + (size_t)h->n_pad * BCM_S;
    bool counting = true;  // the path counts are integers so far
    unsigned long long count_bits = 1ull;
    k_bcm_init<<<grid, 256, 0, st>>>(d, count, dep);
    k_bcm_roots<<<1, BCM_S, 0, st>>>(d, m.roots, kb, count);
    unsigned long long* lf0 = nullptr;
    if ((s = bc_level_word(h, b, 0, &lf0)) != SS_OK) return s;
    k_bcm_keep<<<grid, 256, 0, st>>>(d, m.F[0], W, lf0);
    SS_CUDA(cudaGetLastError());
    if ((s = toc()) != SS_OK) return s;
    // forward: the levels of the batch's sources and their path counts
    int D = 0;
    for (int L = 1;; ++L) {
      if (L > h->n + 1) {
        set_error("slimsell_bc: no convergence after %d levels", L);
        return SS_ERR_CUDA;
      }
      bool done = false;
      if ((s = multi_level(h, m, W, st, &done, kernel_ms ? h->ev_a : nullptr,
                           kernel_ms ? h->ev_b : nullptr)) != SS_OK)
        return s;
      if (kernel_ms) {
        SS_CUDA(cudaEventElapsedTime(&ms, h->ev_a, h->ev_b));
        ms_sum += ms;
      }
      count_bits = h->h_ctl->count_bits;  // read with the level's counters: counts up to level L - 1
      if (done) break;
      if ((s = tic()) != SS_OK) return s;
      if (counting && !bc_counts_fit(count_bits, h->max_degree)) {
        k_bcm_to_fp64<<<grid, 256, 0, st>>>(d, b->sigma);
        counting = false;
      }
      unsigned long long* lfL = nullptr;
      if ((s = bc_level_word(h, b, (size_t)L, &lfL)) != SS_OK) return s;
      k_bcm_keep<<<grid, 256, 0, st>>>(d, m.F[L & 1], W, lfL);
      SS_CUDA(cudaMemsetAsync(&h->ctl->units, 0, sizeof(unsigned long long), st));
      k_bcm_expand<<<grid, 256, 0, st>>>(d, lfL);
      if (counting)
        k_bcm_gather<BC_COUNT><<<grid, 256, 0, st>>>(d, lfL, b->lf[(size_t)L - 1], count, count);
      else
        k_bcm_gather<BC_FP64><<<grid, 256, 0, st>>>(d, lfL, b->lf[(size_t)L - 1], sigma, sigma);
      SS_CUDA(cudaGetLastError());
      if ((s = toc()) != SS_OK) return s;
      D = L;
    }
    if ((s = tic()) != SS_OK) return s;
    // backward: the deepest level has no dependents (delta = 0, t = 1 / sigma)
    if (D >= 1) {
      const int F = bc_fraction_bits(h->n);
      const bool fixed = counting && bc_dependencies_fit(count_bits, F);
      if (counting && !fixed) k_bcm_to_fp64<<<grid, 256, 0, st>>>(d, b->sigma);
      if (!fixed) k_bcm_zero_fp64<<<grid, 256, 0, st>>>(d, sum64);
      for (int L = D; L >= 1; --L) {
        const int leaf = L == D;
        unsigned long long* const lfL = b->lf[(size_t)L];
        if (!leaf) {
          SS_CUDA(cudaMemsetAsync(&h->ctl->units, 0, sizeof(unsigned long long), st));
          k_bcm_expand<<<grid, 256, 0, st>>>(d, lfL);
          if (fixed)
            k_bcm_gather<BC_FIXED><<<grid, 256, 0, st>>>(d, lfL, b->lf[(size_t)L + 1], dep, dep);
          else
            k_bcm_gather<BC_FP64><<<grid, 256, 0, st>>>(d, lfL, b->lf[(size_t)L + 1], t64, sum64);
        }
        if (fixed)
          k_bcm_post_fixed<<<grid, 256, 0, st>>>(d, lfL, count, dep, F, leaf, d_bc);
        else
          k_bcm_post_fp64<<<grid, 256, 0, st>>>(d, lfL, sigma, sum64, t64, leaf, d_bc);
      }
      SS_CUDA(cudaGetLastError());
    }
    if ((s = toc()) != SS_OK) return s;
  }
  SS_CUDA(cudaStreamSynchronize(st));
  if (kernel_ms) *kernel_ms = ms_sum;
  return SS_OK;
}
