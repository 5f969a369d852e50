// Exact selection of the smallest keys of a long array by one thread-block
// cluster (1 to 8 CTAs of 1024 threads): the top-k of the screening pool.
//
// At most three histogram passes over 32-bit keys, 2048 bins each, that narrow
// the range [lo, hi] of the wanted rank: the first over the span between the
// smallest and the largest key.  (Bins of fixed bits put nearly all keys, which
// are close together, into a few: every add then met the same address, and
// merging a warp's equal bins first, with match.any, took 16 of the 29 us of
// 65,536 scores.)  Every CTA counts its own elements into a shared-memory
// histogram, the cluster synchronises, and every CTA adds the histograms of
// all through distributed shared memory and finds the bin of the wanted rank
// by a block scan.  One CTA alone was bound by the latency of its passes over
// the array (64 reads a thread and pass, seven passes: 150 us); eight CTAs
// keep eight keys a thread in registers.
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"

namespace cem {

constexpr int kSelThreads = 1024;
constexpr int kSelBins = 2048;
constexpr int kSelPasses = 3;
constexpr int kSelCtas = 8;  // the largest cluster

// CTAs of the cluster that selects from n keys: one while each thread has at
// most four, then enough to keep eight a thread in registers, up to eight
inline int select_ctas(int n) { return n <= 4 * kSelThreads ? 1 : n <= 16 * kSelThreads ? 4 : kSelCtas; }

// the keys below `key` (which need not be one) and `take` of the `equal` ones
// that equal it are the wanted ones
struct Cut {
  uint32_t key;
  int take, equal;
};

struct SelectShared {
  uint32_t hist[kSelPasses][kSelBins];
  uint32_t warp_sum[32];
  uint2 range;  // smallest and largest key of this CTA
  uint32_t bin, before, in_bin;
};

// order-preserving bits of a float (a negative zero counts as zero)
__device__ __forceinline__ uint32_t float_order(float x) {
  const uint32_t u = __float_as_uint(x + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ void select_clear(SelectShared& sh) {
  for (int i = threadIdx.x; i < kSelPasses * kSelBins; i += kSelThreads) (&sh.hist[0][0])[i] = 0u;
}

// inclusive scan over the block; tot: a 32-entry array in shared memory (used
// by this call alone until the next __syncthreads)
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* tot) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) tot[w] = x;
  __syncthreads();
  uint32_t t = tot[lane];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += y;
  }
  const uint32_t before = __shfl_sync(0xffffffffu, t, w > 0 ? w - 1 : 0);
  return x + (w > 0 ? before : 0u);
}

// The `need` smallest keys (need >= 1, at most the number of valid keys).
// each(f) calls f(valid, key) for this thread's elements.  The histograms have
// been cleared (select_clear and a __syncthreads).  All threads of the cluster
// take part and get the result.
template <class Each>
__device__ __forceinline__ Cut cluster_select(cooperative_groups::cluster_group& cl, SelectShared& sh, Each each,
                                              uint32_t need) {
  const int tid = threadIdx.x, lane = tid & 31, nc = (int)cl.num_blocks();
  uint32_t lo = 0xffffffffu, hi = 0u, equal = 0u;
  each([&](bool valid, uint32_t key) {
    if (valid) {
      lo = min(lo, key);
      hi = max(hi, key);
    }
  });
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {  // (the third pass's histogram is free until then)
    sh.hist[kSelPasses - 1][tid >> 5] = lo;
    sh.hist[kSelPasses - 1][32 + (tid >> 5)] = hi;
  }
  __syncthreads();
  lo = __reduce_min_sync(0xffffffffu, sh.hist[kSelPasses - 1][lane]);
  hi = __reduce_max_sync(0xffffffffu, sh.hist[kSelPasses - 1][32 + lane]);
  if (tid == 0) sh.range = make_uint2(lo, hi);
  __syncthreads();
  if (tid < 64) sh.hist[kSelPasses - 1][tid] = 0u;
  if (nc > 1) {
    cl.sync();
#pragma unroll
    for (int r = 0; r < kSelCtas; ++r)
      if (r < nc) {
        const uint2 q = *cl.map_shared_rank(&sh.range, r);
        lo = min(lo, q.x);
        hi = max(hi, q.y);
      }
  } else {
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < kSelPasses; ++p) {
    const int bits = 32 - __clz(hi - lo), shift = bits > 11 ? bits - 11 : 0;
    each([&](bool valid, uint32_t key) {
      if (valid && key >= lo && key <= hi) atomicAdd(&sh.hist[p][CEM_DIDX((key - lo) >> shift, kSelBins, 12)], 1u);
    });
    if (nc > 1) cl.sync();
    else __syncthreads();
    uint32_t a = 0, b = 0;
    if (nc > 1) {  // (unrolled: the remote reads are in flight together)
#pragma unroll
      for (int r = 0; r < kSelCtas; ++r)
        if (r < nc) {
          const uint2 h = *reinterpret_cast<const uint2*>(cl.map_shared_rank(&sh.hist[p][0], r) + 2 * tid);
          a += h.x;
          b += h.y;
        }
    } else {
      a = sh.hist[p][2 * tid];
      b = sh.hist[p][2 * tid + 1];
    }
    const uint32_t incl = block_scan(a + b, sh.warp_sum), excl = incl - a - b;
    if (excl < need && need <= incl) {
      const bool second = need > excl + a;
      sh.bin = (uint32_t)(2 * tid) + (second ? 1u : 0u);
      sh.before = excl + (second ? a : 0u);
      sh.in_bin = second ? b : a;
    }
    __syncthreads();
    lo += sh.bin << shift;
    hi = min(hi, lo + ((1u << shift) - 1u));
    need -= sh.before;
    equal = sh.in_bin;
    __syncthreads();
    // (these are the same in every thread of the cluster)
    if (shift == 0) break;
    if (need == equal) return Cut{hi + 1u, 0, 0};  // the whole bin is wanted (usually after two passes)
  }
  return Cut{lo, (int)need, (int)equal};
}

}  // namespace cem
