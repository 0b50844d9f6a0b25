// Pieces of the pull kernels (single- and multi-source): streaming column loads and
// the shared-memory image of a row bitmap.
#pragma once

#include "ss_device.cuh"

namespace ss {

#ifndef SS_PULL_LOAD
#define SS_PULL_LOAD 2  // col loads: 0 evict-first, 1 no-L1 with 256-byte L2 fetches, 2 no-L1
#endif

// Stage the bitmap prefix only when the previous iteration read at least this
// many slots; below it, reading frontier bits from global memory is cheaper.
constexpr unsigned long long STAGE_MIN_SLOTS = 2ull << 20;

__device__ __forceinline__ int4 ld_stream(const int4* p) {
#if SS_PULL_LOAD == 1
  int4 v;
  asm("ld.global.nc.L1::no_allocate.L2::256B.v4.s32 {%0, %1, %2, %3}, [%4];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p));
  return v;
#elif SS_PULL_LOAD == 2
  int4 v;
  asm("ld.global.nc.L1::no_allocate.v4.s32 {%0, %1, %2, %3}, [%4];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p));
  return v;
#else
  return __ldcs(p);
#endif
}

extern __shared__ __align__(16) unsigned ss_smem_bits[];

// Shared-memory image of the bitmap: SMEM_GUARD zero words, then the staged
// prefix.  The padding marker c = -1 has c >> 5 = -1 and lands on the last guard
// word, so it needs no branch; vertices past the prefix read the global bitmap.
constexpr int SMEM_GUARD = 4;

__device__ __forceinline__ unsigned frontier_bit(const unsigned* smw, int sbits, const unsigned* gbm,
                                                 int c) {
  const int wi = c >> 5;
  const unsigned w = (c < sbits) ? smw[wi] : __ldg(gbm + wi);
  return (w >> (c & 31)) & 1u;
}

// Store the C frontier bits of one chunk (bit l = row l) into the bitmap.
template <int C>
__device__ __forceinline__ void store_bits(unsigned* fb, int chunk, unsigned lo, unsigned hi) {
  if (C == 8) reinterpret_cast<unsigned char*>(fb)[chunk] = (unsigned char)lo;
  else if (C == 16) reinterpret_cast<unsigned short*>(fb)[chunk] = (unsigned short)lo;
  else if (C == 32) fb[chunk] = lo;
  else reinterpret_cast<uint2*>(fb)[chunk] = make_uint2(lo, hi);
}

// Start copying the first `words` bitmap words (a multiple of 4) behind the guard;
// returns the shared address of the first one.
__device__ __forceinline__ unsigned stage_words(const unsigned* gbm, int words) {
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(ss_smem_bits + SMEM_GUARD);
  for (int i = threadIdx.x; i < (words >> 2); i += blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sbase + 16u * (unsigned)i),
                 "l"(reinterpret_cast<const int4*>(gbm) + i)
                 : "memory");
  return sbase;
}

__device__ __forceinline__ void stage_wait() {
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
}

}  // namespace ss
