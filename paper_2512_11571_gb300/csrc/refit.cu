// Update step of Algorithm 1 (Sec. III-B): pick the top-N_e elites and refit
// the sampling distribution to them.
//
// Elite rules of Sec. III-B: samples are ranked by (class, J, index); the
// elites are the K lowest of the best class present among {0: goal reached,
// 1: every action succeeded} -- fewer if fewer exist ("only the n_feasible
// samples are used") -- or, if neither class occurs, of class 2.  The new
// distribution is the maximum-likelihood Gaussian of the elites (the
// KL-minimising CE update of Botev et al.): mean, covariance with 1/K_eff,
// a ridge (1e-4 range)^2; a single elite gets diag((0.05 range)^2)
// ("artificial noise"); the diagonal mode is the independent-normal model of
// Sec. IV-A.
//
// One CTA of 1024 threads per problem.  Selection is exact: a radix select
// over the span of the class's costs (order-preserving 32-bit keys; 2048 bins a
// pass, at most three passes, and it ends as soon as a whole bin is wanted), and
// of costs equal to the last one wanted, those with the lowest indices.  The
// keys of the first KR * 1024 samples stay in registers across the passes.  The
// K_eff elites (<= 4096 keys of cost and index in shared memory) are then
// sorted, up to 1024 of them with one key in each thread's register.  Up to 512
// samples are ranked by counting instead.  The
// statistics are accumulated in FP64 by groups of four threads per output with
// a fixed reduction order: with few elites the covariance hangs on its ridge,
// the last bit of a sum shows in the factor, and a CE run that follows it parts
// from its earlier self.  One warp factorises the covariance.
//
// Bound by the latency of one CTA's chain of barriers, and for many elites by
// its FP64 pipe (K = 512, D = 14: 68,000 operations at two a cycle).  Refit and
// next draw of N = 16384, K = 512, D = 14: 67 us; 95 us with seven passes of
// fixed 8-bit digits over 52-bit keys, merged per warp by match.any, four
// samples a thread in registers, the sort through shared memory and a row per
// lane in the factorisation.  A search of N = 256, K = 25, ten iterations: 704
// us, 717 before; 723 with the radix select at that size too.
#include "internal.h"
#include "select.cuh"

namespace cem {
namespace {

constexpr int RT = kSelThreads;
constexpr int KR = 16;  // samples per thread whose keys stay in registers (N <= 16,384 entirely)
// up to this many samples are ranked by counting the smaller keys (2 us an
// iteration less than the radix select and the sort at 256; the count grows
// with N^2: at 1024 it is 32,000 shared-memory reads of a warp)
constexpr int KCOUNT = 512;
constexpr uint32_t kNoKey = 0xffffffffu;  // above every finite cost's key
// up to this many elites are staged in shared memory as FP64 rows for the
// statistics (18 parameters: 72 KB); more are read through L2
constexpr int KSTAGE = 512;

// class (0..3) and order-preserving cost bits of sample i (a cost that is not
// finite: class 3)
__device__ __forceinline__ int classify(const float* __restrict__ J, const uint8_t* __restrict__ cls, int i,
                                        uint32_t& key) {
  const float j = J[i];
  const int c = isfinite(j) ? min((int)cls[i], 3) : 3;
  key = float_order(j);
  return c;
}

// The `need` smallest keys (1 <= need <= number of keys that are not kNoKey).
// each(f) calls f(key) for this thread's elements.
template <class Each>
__device__ __forceinline__ Cut block_select(SelectShared& sh, Each each, uint32_t need) {
  const int tid = threadIdx.x, lane = tid & 31;
  __syncthreads();  // (an earlier selection may still be read)
  select_clear(sh);
  uint32_t lo = kNoKey, hi = 0u;
  each([&](uint32_t key) {
    if (key != kNoKey) {
      lo = min(lo, key);
      hi = max(hi, key);
    }
  });
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (tid == 0) sh.range = make_uint2(kNoKey, 0u);
  __syncthreads();
  if (lane == 0) {
    atomicMin(&sh.range.x, lo);
    atomicMax(&sh.range.y, hi);
  }
  __syncthreads();
  lo = sh.range.x;
  hi = sh.range.y;
  uint32_t equal = 0u;
#pragma unroll 1
  for (int p = 0; p < kSelPasses; ++p) {
    const int bits = 32 - __clz(hi - lo), shift = bits > 11 ? bits - 11 : 0;
    each([&](uint32_t key) {
      if (key != kNoKey && key >= lo && key <= hi) atomicAdd(&sh.hist[p][CEM_DIDX((key - lo) >> shift, kSelBins, 12)], 1u);
    });
    __syncthreads();
    const uint32_t a = sh.hist[p][2 * tid], b = sh.hist[p][2 * tid + 1];
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
    // (these are the same in every thread)
    if (shift == 0) break;
    if (need == equal) return Cut{hi + 1u, 0, 0};  // the whole bin is wanted
  }
  return Cut{lo, (int)need, (int)equal};
}

// ascending bitonic sort of P (a power of two) keys in shared memory; up to RT
// of them with one in each thread's register, exchanged by shuffles inside a
// warp
__device__ __forceinline__ void sort_keys(uint64_t* keys, int P) {
  const int tid = threadIdx.x;
  if (P <= RT) {
    const bool in = tid < P;
    uint64_t x = in ? keys[tid] : ~0ull;
    for (int k = 2; k <= P; k <<= 1) {
      const bool asc = (tid & k) == 0;
      for (int j = k >> 1; j > 0; j >>= 1) {
        uint64_t y;
        if (j >= 32) {
          __syncthreads();
          if (in) keys[tid] = x;
          __syncthreads();
          y = in ? keys[tid ^ j] : ~0ull;
        } else {
          y = __shfl_xor_sync(0xffffffffu, x, j);
        }
        const bool low = (tid & j) == 0;  // this thread keeps the smaller one of an ascending pair
        if ((x > y) == (low == asc)) x = y;
      }
    }
    __syncthreads();
    if (in) keys[tid] = x;
    __syncthreads();
    return;
  }
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = tid; i < P; i += RT) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const uint64_t x = keys[i], y = keys[ixj];
          const bool asc = (i & k) == 0;
          if ((x > y) == asc) {
            keys[i] = y;
            keys[ixj] = x;
          }
        }
      }
      __syncthreads();
    }
}

// right-looking Cholesky factor in place, lower triangle, by one warp: the
// trailing update of a column is spread over the lanes element by element
// (with a row per lane, one row's chain of updates took 1800 cycles a column
// at D = 14).  tri[t] = 32 p + q for t = p (p + 1) / 2 + q, q <= p
constexpr int kTri = (CEM_MAX_D - 1) * CEM_MAX_D / 2;
__device__ bool cholesky_warp(double* A, int D, int lane, const uint16_t* tri) {
  for (int j = 0; j < D; ++j) {
    const double d = A[j * D + j];
    if (!__all_sync(0xffffffffu, d > 0.0)) return false;
    // one reciprocal square root instead of a square root and a division
    // per row (FP64 is slow on this part; the result is cast to FP32)
    const double r = rsqrt(d);
    const double ljj = d * r;
    __syncwarp();
    if (lane == j) A[j * D + j] = ljj;
    if (lane > j && lane < D) A[lane * D + j] *= r;
    __syncwarp();
    // elements (j + 1 + p, j + 1 + q), q <= p, of the trailing triangle
    const int m = D - 1 - j;
    for (int t = lane; t < m * (m + 1) / 2; t += 32) {
      const int i = j + 1 + (tri[t] >> 5), k = j + 1 + (tri[t] & 31);
      A[i * D + k] = fma(-A[i * D + j], A[k * D + j], A[i * D + k]);
    }
    __syncwarp();
  }
  return true;
}

__device__ __forceinline__ void refit_body(const RefitArgs& a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ SelectShared sh;
  __shared__ int cnt[4];
  __shared__ int s_n, s_fail;
  __shared__ double s_mean[CEM_MAX_D];
  __shared__ double s_cov[CEM_MAX_D * CEM_MAX_D];
  __shared__ double s_L[CEM_MAX_D * CEM_MAX_D];
  __shared__ uint16_t s_tri[kTri];
  const int tid = threadIdx.x, lane = tid & 31, N = a.N, D = a.D;
  if (tid < 4) cnt[tid] = 0;
  if (tid == 0) s_n = 0;
  if (const int t = RT - 1 - tid; t < kTri) {  // (the last warps: they have the fewest samples)
    int p = 0;
    while ((p + 1) * (p + 2) / 2 <= t) ++p;
    s_tri[t] = (uint16_t)(32 * p + t - p * (p + 1) / 2);
  }
  __syncthreads();
  // keys and classes (two bits each) of samples tid + r * RT, r < KR
  uint32_t rkey[KR], rcls = 0u;
  {
    int n0 = 0, n1 = 0, n2 = 0, n3 = 0;
    auto count = [&](int c) {
      n0 += c == 0;
      n1 += c == 1;
      n2 += c == 2;
      n3 += c == 3;
    };
#pragma unroll
    for (int r = 0; r < KR; ++r) {
      const int i = r * RT + tid;
      rkey[r] = kNoKey;
      if (i < N) {
        const int c = classify(a.J, a.cls, i, rkey[r]);
        rcls |= (uint32_t)c << (2 * r);
        count(c);
      }
    }
    for (int i = KR * RT + tid; i < N; i += RT) {
      uint32_t key;
      count(classify(a.J, a.cls, i, key));
    }
    n0 = __reduce_add_sync(0xffffffffu, n0);
    n1 = __reduce_add_sync(0xffffffffu, n1);
    n2 = __reduce_add_sync(0xffffffffu, n2);
    n3 = __reduce_add_sync(0xffffffffu, n3);
    if (lane < 4) {
      const int n = lane == 0 ? n0 : lane == 1 ? n1 : lane == 2 ? n2 : n3;
      if (n) atomicAdd(&cnt[lane], n);
    }
  }
  __syncthreads();
  const int cstar = cnt[0] > 0 ? 0 : cnt[1] > 0 ? 1 : cnt[2] > 0 ? 2 : -1;
  const int in_class = cstar < 0 ? 0 : cnt[cstar];
  const int keff = min(a.K, in_class);
  if (keff > 0) {
    // kNoKey for the samples of other classes
#pragma unroll
    for (int r = 0; r < KR; ++r)
      if ((int)((rcls >> (2 * r)) & 3u) != cstar) rkey[r] = kNoKey;
    auto each = [&](auto f) {  // f(sample, key), whole warps together
#pragma unroll
      for (int r = 0; r < KR; ++r)
        if (r * RT < N) f(r * RT + tid, rkey[r]);
      for (int base = KR * RT; base < N; base += RT) {
        const int i = base + tid;
        uint32_t key = kNoKey;
        if (i < N && classify(a.J, a.cls, i, key) != cstar) key = kNoKey;
        f(i, key);
      }
    };
    int P = 1;
    while (P < keff) P <<= 1;
    uint64_t* keys = reinterpret_cast<uint64_t*>(dyn);
    if (N <= KCOUNT) {
      // RT / Pn threads count the keys below each sample's
      int Pn = 32;
      while (Pn < N) Pn <<= 1;
      uint64_t* all = reinterpret_cast<uint64_t*>(&sh.hist[0][0]);
      uint32_t* rank = &sh.hist[1][0];
      if (tid < Pn) {
        all[tid] = rkey[0] != kNoKey ? ((uint64_t)rkey[0] << 20) | (uint64_t)tid : ~0ull;
        rank[tid] = 0u;
      }
      __syncthreads();
      const int e = tid & (Pn - 1), parts = RT / Pn;
      const uint64_t key = all[e];
      uint32_t below = 0u;
      if (key != ~0ull) {
#pragma unroll 4
        for (int q = tid / Pn; q < N; q += parts) below += all[q] < key;
        atomicAdd(&rank[e], below);
      }
      __syncthreads();
      if (tid < Pn && key != ~0ull && rank[tid] < (uint32_t)keff) keys[rank[tid]] = key;
      __syncthreads();
    } else {
      // elites: costs below the cut, and of those equal to it the ones of samples
      // before tie_end
      Cut cut{kNoKey, 0, 0};
      uint32_t tie_end = 0u;
      if (keff < in_class) {
        cut = block_select(sh, [&](auto f) { each([&](int, uint32_t key) { f(key); }); }, (uint32_t)keff);
        if (cut.take > 0) {
          tie_end = kNoKey;
          if (cut.take < cut.equal) {
            const Cut t = block_select(sh, [&](auto f) {
              each([&](int i, uint32_t key) { f(key == cut.key ? (uint32_t)i : kNoKey); });
            }, (uint32_t)cut.take);
            tie_end = t.key + (t.take > 0 ? 1u : 0u);
          }
        }
      }
      // gather the elites (unordered), then bitonic sort by key
      for (int i = tid; i < P; i += RT) keys[i] = ~0ull;
      __syncthreads();
      each([&](int i, uint32_t key) {
        const bool in = key < cut.key || (key == cut.key && key != kNoKey && (uint32_t)i < tie_end);
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (m == 0u) return;
        int pos = 0;
        if (lane == __ffs(m) - 1) pos = atomicAdd(&s_n, __popc(m));
        pos = __shfl_sync(0xffffffffu, pos, __ffs(m) - 1) + __popc(m & ((1u << lane) - 1u));
        if (in && pos < P) keys[pos] = ((uint64_t)key << 20) | (uint64_t)i;
      });
      __syncthreads();
      sort_keys(keys, P);
    }
    if (a.elite_idx)
      for (int e = tid; e < keff; e += RT) a.elite_idx[e] = CEM_DIDX((int)(keys[e] & 0xFFFFF), a.N, 8);
    // elite e's parameter row (read through L2; the keys stay in shared memory)
    auto eth = [&](int e, int d) -> float { return a.theta[(size_t)CEM_DIDX((int)(keys[e] & 0xFFFFF), a.N, 8) * D + d]; };
    // statistics in FP64: 4 threads per output, fixed reduction order
    const int grp = tid >> 2, part = tid & 3;
    const double invk = 1.0 / (double)keff;
    if (keff == 1) {
      if (tid < D) s_mean[tid] = (double)eth(0, tid);
      for (int i = tid; i < D * D; i += RT) {
        const int r = i / D, c = i % D;
        const double w = 0.05 * ((double)a.hi[r] - (double)a.lo[r]);
        s_cov[i] = r == c ? w * w : 0.0;
      }
      __syncthreads();
    } else {
      // keff <= KSTAGE: the elite rows once into shared memory (X[e][d] as
      // FP64), centred after the mean, so each covariance term is one FP64
      // multiply-add on shared operands; the sums run in the same order and
      // give the same values as the L2 path
      const bool staged = keff <= KSTAGE;
      double* X = reinterpret_cast<double*>(dyn + sizeof(uint64_t) * (size_t)P);
      if (staged) {
        for (int q = tid; q < keff * D; q += RT) {
          const int e = q / D;
          X[q] = (double)eth(e, q - e * D);
        }
        __syncthreads();
      }
      double v = 0.0;
      if (grp < D) {
        if (staged)
          for (int e = part; e < keff; e += 4) v += X[e * D + grp];
        else
          for (int e = part; e < keff; e += 4) v += (double)eth(e, grp);
      }
      v += __shfl_down_sync(0xffffffffu, v, 2);
      v += __shfl_down_sync(0xffffffffu, v, 1);
      if (grp < D && part == 0) s_mean[grp] = v * invk;
      __syncthreads();
      if (staged) {
        for (int q = tid; q < keff * D; q += RT) X[q] -= s_mean[q % D];
        __syncthreads();
      }
      const int npair = D * (D + 1) / 2;
      int pi = 0, pj = 0;
      if (grp < npair) {  // pair index -> (pi, pj), pi <= pj
        int rem = grp, r = 0;
        while (rem >= D - r) {
          rem -= D - r;
          ++r;
        }
        pi = r;
        pj = r + rem;
      }
      v = 0.0;
      if (grp < npair) {
        if (staged) {
          for (int e = part; e < keff; e += 4) v += X[e * D + pi] * X[e * D + pj];
        } else {
          const double mi = s_mean[pi], mj = s_mean[pj];
          for (int e = part; e < keff; e += 4) v += ((double)eth(e, pi) - mi) * ((double)eth(e, pj) - mj);
        }
      }
      v += __shfl_down_sync(0xffffffffu, v, 2);
      v += __shfl_down_sync(0xffffffffu, v, 1);
      if (grp < npair && part == 0) {
        double c = v * invk;
        if (pi == pj) {
          const double w = 1e-4 * ((double)a.hi[pi] - (double)a.lo[pi]);
          c += w * w;
        }
        s_cov[pi * D + pj] = c;
        s_cov[pj * D + pi] = c;
      }
      __syncthreads();
    }
    if (a.cov_mode == CEM_COV_DIAG)
      for (int i = tid; i < D * D; i += RT)
        if (i / D != i % D) s_cov[i] = 0.0;
    __syncthreads();
    if (tid < 32) {
      for (int i = tid; i < D * D; i += 32) s_L[i] = (i % D) <= (i / D) ? s_cov[i] : 0.0;
      __syncwarp();
      bool ok = cholesky_warp(s_L, D, tid, s_tri);
      if (!ok) {  // fall back to the diagonal
        for (int i = tid; i < D * D; i += 32) {
          const bool dg = i / D == i % D;
          if (!dg) s_cov[i] = 0.0;
          s_L[i] = dg ? s_cov[i] : 0.0;
        }
        __syncwarp();
        ok = cholesky_warp(s_L, D, tid, s_tri);
      }
      if (tid == 0) s_fail = ok ? 0 : 1;
    }
    __syncthreads();
    if (!s_fail) {
      for (int i = tid; i < D; i += RT) a.mean[i] = (float)s_mean[i];
      for (int i = tid; i < D * D; i += RT) {
        a.cov[i] = (float)s_cov[i];
        a.chol[i] = (i % D) <= (i / D) ? (float)s_L[i] : 0.0f;
      }
    } else if (tid == 0 && a.status) {
      *a.status = CEM_ERR_NOT_PD;
    }
  }
  if (tid == 0) {
    if (a.k_eff) *a.k_eff = keff;
    if (a.track) {
      Track* t = a.track;
      if (keff > 0) {
        const int b = CEM_DIDX((int)(reinterpret_cast<uint64_t*>(dyn)[0] & 0xFFFFF), a.N, 8);
        const float jb = a.J[b];
        if (cstar < t->best_cls || (cstar == t->best_cls && jb < t->best_J)) {
          t->best_cls = cstar;
          t->best_J = jb;
          for (int d = 0; d < D; ++d) t->best_theta[d] = a.theta[(size_t)b * D + d];
        }
      }
      const int h = (int)(t->iter - t->base_iter);
      if (h >= 0 && h < t->hist_len) {
        if (a.hist_J) a.hist_J[h] = t->best_J;
        if (a.hist_keff) a.hist_keff[h] = keff;
        if (a.hist_cnt)
          for (int c = 0; c < 4; ++c) a.hist_cnt[4 * h + c] = cnt[c];
      }
      t->iter += 1;
    }
  }
}

__global__ void __launch_bounds__(RT) refit_kernel(RefitArgs a) { refit_body(a); }

// one CTA per problem of a batch; args[p] describes problem p
__global__ void __launch_bounds__(RT) refit_batch_kernel(const RefitArgs* __restrict__ args) {
  __shared__ RefitArgs a;
  if (threadIdx.x == 0) a = args[blockIdx.x];
  __syncthreads();
  if (a.skip) return;  // an eliminated plan keeps its state
  refit_body(a);
}

}  // namespace

#ifdef CEM_DEBUG
CEM_DEBUG_STATUS_ACCESSOR(debug_status_refit)
#endif

size_t refit_smem_bytes(int K, int D) {
  int P = 1;
  while (P < K) P <<= 1;
  const int ks = K < KSTAGE ? K : KSTAGE;
  return sizeof(uint64_t) * (size_t)P + sizeof(double) * (size_t)(ks > 0 ? ks : 0) * (size_t)(D > 0 ? D : 0);
}

cudaError_t configure_refit() {
  cudaError_t e = cudaFuncSetAttribute(refit_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)refit_smem_bytes(CEM_MAX_K, CEM_MAX_D));
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(refit_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)refit_smem_bytes(CEM_MAX_K, CEM_MAX_D));
}

cudaError_t launch_refit_batch(const RefitArgs* args_d, int n_problems, int maxK, int maxD, cudaStream_t st) {
  if (n_problems <= 0) return cudaSuccess;
  refit_batch_kernel<<<n_problems, RT, refit_smem_bytes(maxK, maxD), st>>>(args_d);
  return cudaGetLastError();
}

cudaError_t launch_refit(const RefitArgs& a, cudaStream_t st) {
  refit_kernel<<<1, RT, refit_smem_bytes(a.K, a.D), st>>>(a);
  return cudaGetLastError();
}

}  // namespace cem
