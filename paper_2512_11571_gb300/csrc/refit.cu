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
// One thread-block cluster of 1, 4 or 8 CTAs of 1024 threads per problem (by
// N, see select_ctas).  Selection is exact: a radix select over the 32-bit
// order-preserving cost bits of the chosen class (select.cuh), one over the
// indices where the cut goes through equal costs, then a bitonic sort of the
// K_eff elites by (cost, index); up to 512 samples are instead ranked by
// counting, which selects and sorts at once.  The statistics are accumulated
// in FP64, a warp per output in a fixed order that does not depend on the
// cluster (run-to-run and batch-to-single identical), the outputs split over
// the CTAs, and one warp of the first CTA factorises the covariance.
//
// What bounds it: latency, and the FP64 units for the statistics (about two
// multiply-adds per cycle and SM: 105 sums of 512 at D = 14 are 27,000 cycles
// in one CTA).  N = 16384, K = 512, D = 14 in one CTA, seven 8-bit passes with
// match.any, one FP64 sum per four threads: 90 us (ncu, cold); here 47 us.
#include "internal.h"
#include "select.cuh"

namespace cem {
namespace {

namespace cg = cooperative_groups;

constexpr int RT = kSelThreads;
constexpr int KR = 8;  // samples per thread whose keys stay in registers
// up to this many samples are ranked by counting (N^2 comparisons over the
// block: 3 us at 512, more than the radix select takes beyond)
constexpr int KCOUNT = 512;
// up to this many elites are staged in shared memory as FP64 columns for the
// statistics (18 parameters: 72 KB); more are read through L2
constexpr int KSTAGE = 512;

// class (0..3) and order-preserving cost bits of sample i (a cost that is not
// finite: class 3, last)
__device__ __forceinline__ int classify(const float* __restrict__ J, const uint8_t* __restrict__ cls, int i,
                                        uint32_t& key) {
  float j = J[i];
  int c = cls[i];
  if (c > 3) c = 3;
  if (!isfinite(j)) {
    c = 3;
    j = __int_as_float(0x7f800000);
  }
  key = float_order(j);
  return c;
}

__device__ __forceinline__ uint64_t elite_key(uint32_t key, int i) { return ((uint64_t)key << 20) | (uint64_t)i; }

// right-looking Cholesky factor in place, lower triangle, by one warp: the
// trailing update of a column is spread over the lanes element by element
// (a row per lane left the chain of one row's updates, 1800 cycles a column
// at D = 14)
// (tri[t] = 32 p + q for t = p (p + 1) / 2 + q, q <= p)
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
      A[i * D + k] -= A[i * D + j] * A[k * D + j];
    }
    __syncwarp();
  }
  return true;
}

// ascending bitonic sort of P (a power of two) keys in shared memory; up to
// RT of them with one in each thread's register, exchanged by shuffles
// inside a warp
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

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void refit_body(const RefitArgs& a) {
  extern __shared__ __align__(16) unsigned char dyn[];
  cg::cluster_group cl = cg::this_cluster();
  __shared__ SelectShared sh;
  __shared__ int cnt[4];
  __shared__ int s_n, s_fail;
  __shared__ double s_mean[CEM_MAX_D];
  __shared__ double s_cov[CEM_MAX_D * CEM_MAX_D];
  __shared__ double s_L[CEM_MAX_D * CEM_MAX_D];
  __shared__ uint16_t s_tri[kTri];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, N = a.N, D = a.D;
  const int nc = (int)cl.num_blocks(), c = (int)cl.block_rank();
  auto sync_all = [&]() {
    if (nc > 1) cl.sync();
    else __syncthreads();
  };
  auto at0 = [&](auto* p) { return nc > 1 ? cl.map_shared_rank(p, 0) : p; };  // the first CTA's copy
  if (tid < 4) cnt[tid] = 0;
  if (tid == 0) s_n = 0;
  select_clear(sh);
  if (tid < kTri) {
    int p = 0;
    while ((p + 1) * (p + 2) / 2 <= tid) ++p;
    s_tri[tid] = (uint16_t)(32 * p + tid - p * (p + 1) / 2);
  }
  __syncthreads();
  // this CTA's samples: c, c + nc, ... in runs of 1024; their keys and classes
  // (4: no sample), the first KR rounds in registers
  const int rounds = (N + nc * RT - 1) / (nc * RT);
  auto index = [&](int r) { return (r * nc + c) * RT + tid; };
  auto sample = [&](int r, uint32_t& key) {
    const int i = index(r);
    key = 0;
    return i < N ? classify(a.J, a.cls, i, key) : 4;
  };
  uint32_t rkey[KR];
  int rcls[KR];
#pragma unroll
  for (int r = 0; r < KR; ++r) {
    rkey[r] = 0;
    rcls[r] = r < rounds ? sample(r, rkey[r]) : 4;
  }
  auto each = [&](auto f) {  // f(index, class, key), whole warps together
#pragma unroll
    for (int r = 0; r < KR; ++r)
      if (r < rounds) f(index(r), rcls[r], rkey[r]);
    for (int r = KR; r < rounds; ++r) {
      uint32_t key;
      const int k = sample(r, key);
      f(index(r), k, key);
    }
  };
  {
    int n0 = 0, n1 = 0, n2 = 0, n3 = 0;
    each([&](int, int k, uint32_t) {
      n0 += k == 0;
      n1 += k == 1;
      n2 += k == 2;
      n3 += k == 3;
    });
    n0 = __reduce_add_sync(0xffffffffu, n0);
    n1 = __reduce_add_sync(0xffffffffu, n1);
    n2 = __reduce_add_sync(0xffffffffu, n2);
    n3 = __reduce_add_sync(0xffffffffu, n3);
    if (lane < 4) {
      const int n = lane == 0 ? n0 : lane == 1 ? n1 : lane == 2 ? n2 : n3;
      if (n) atomicAdd(&cnt[lane], n);
    }
  }
  sync_all();
  int total[4] = {0, 0, 0, 0};
  if (nc > 1) {
#pragma unroll
    for (int r = 0; r < kSelCtas; ++r)
      if (r < nc) {
        const int* q = cl.map_shared_rank(&cnt[0], r);
#pragma unroll
        for (int k = 0; k < 4; ++k) total[k] += q[k];
      }
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) total[k] = cnt[k];
  }
  const int cstar = total[0] > 0 ? 0 : total[1] > 0 ? 1 : total[2] > 0 ? 2 : -1;
  const int in_class = cstar == 0 ? total[0] : cstar == 1 ? total[1] : cstar == 2 ? total[2] : 0;
  const int keff = min(a.K, in_class);
  uint64_t* keys = reinterpret_cast<uint64_t*>(dyn);
  if (keff > 0) {
    int P = 1;
    while (P < keff) P <<= 1;
    if (nc == 1 && N <= KCOUNT) {
      // every key of the class in shared memory; a sample's rank is the number
      // of smaller keys (counted by RT / 512 threads per sample)
      uint64_t* all = reinterpret_cast<uint64_t*>(&sh.hist[0][0]);
      const uint64_t mine = rcls[0] == cstar ? elite_key(rkey[0], tid) : ~0ull;
      if (tid < KCOUNT) all[tid] = mine;
      __syncthreads();
      const int e = tid & (KCOUNT - 1), half = tid / KCOUNT;
      const uint64_t key = all[e];
      int rank = 0;
      if (e < N)
#pragma unroll 4
        for (int q = half; q < N; q += RT / KCOUNT) rank += all[q] < key;
      int* part = reinterpret_cast<int*>(&sh.hist[1][0]);
      if (half) part[e] = rank;
      __syncthreads();
      if (!half) {
        rank += part[e];
        if (key != ~0ull && rank < keff) keys[rank] = key;
      }
      __syncthreads();
    } else {
      Cut cut{0xffffffffu, 0, 0};
      uint32_t tie_end = 0xffffffffu;  // samples of the cut's cost up to this index (exclusive)
      if (keff < in_class) {
        cut = cluster_select(cl, sh, [&](auto f) { each([&](int, int k, uint32_t key) { f(k == cstar, key); }); },
                             (uint32_t)keff);
        if (cut.take < cut.equal) {  // of equal costs, those with the lowest indices
          sync_all();
          select_clear(sh);
          __syncthreads();
          const Cut t = cluster_select(cl, sh, [&](auto f) {
            each([&](int i, int k, uint32_t key) { f(k == cstar && key == cut.key, (uint32_t)i); });
          }, (uint32_t)cut.take);
          tie_end = t.key + (t.take > 0 ? 1u : 0u);
        }
      }
      // gather the elites (unordered), then sort them: in a cluster every CTA
      // gets all of them and ranks its share by counting, a single CTA (or more
      // than 1024 elites) sorts them in the first one
      const bool count = nc > 1 && keff <= RT;
      uint64_t* bag = count ? reinterpret_cast<uint64_t*>(&sh.hist[0][0]) : keys;
      if (!count && c == 0)
        for (int i = tid; i < P; i += RT) keys[i] = ~0ull;
      sync_all();  // (nobody reads this CTA's histograms any more)
      int* n0 = at0(&s_n);
      uint64_t* bag0 = at0(bag);
      each([&](int i, int k, uint32_t key) {
        const bool in = k == cstar && (key < cut.key || (key == cut.key && (uint32_t)i < tie_end));
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (m == 0u) return;
        int pos = 0;
        if (lane == __ffs(m) - 1) pos = atomicAdd(n0, __popc(m));
        pos = __shfl_sync(0xffffffffu, pos, __ffs(m) - 1) + __popc(m & ((1u << lane) - 1u));
        if (in && pos < P) {
          if (count)
            for (int r = 0; r < nc; ++r) cl.map_shared_rank(bag, r)[pos] = elite_key(key, i);
          else
            bag0[pos] = elite_key(key, i);
        }
      });
      sync_all();
      if (count) {
        const int per = (keff + nc - 1) / nc;  // elites e = c per .. of this CTA, tpk threads each
        int tpk = 32;
        while (tpk * per > RT) tpk >>= 1;
        const int e = c * per + tid / tpk;
        const bool mine = tid / tpk < per && e < keff;
        const uint64_t key = mine ? bag[e] : 0ull;
        int rank = 0;
        if (mine)
#pragma unroll 8
          for (int q = tid & (tpk - 1); q < keff; q += tpk) rank += bag[q] < key;
        for (int o = tpk >> 1; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        if (mine)
          for (int r = tid & (tpk - 1); r < nc; r += tpk) cl.map_shared_rank(keys, r)[rank] = key;
        cl.sync();
      } else {
        if (c == 0) sort_keys(keys, P);
        if (nc > 1) {  // every CTA takes the sorted keys
          cl.sync();
          if (c > 0)
            for (int i = tid; i < keff; i += RT) keys[i] = bag0[i];
          __syncthreads();
        }
      }
    }
    if (c == 0 && a.elite_idx)
      for (int e = tid; e < keff; e += RT) a.elite_idx[e] = (int)(keys[e] & 0xFFFFF);
    // elite e's parameter row (read through L2; the keys stay in shared memory)
    auto eth = [&](int e, int d) -> float { return a.theta[(size_t)CEM_DIDX((int)(keys[e] & 0xFFFFF), a.N, 8) * D + d]; };
    double* mean0 = at0(s_mean);
    double* cov0 = at0(s_cov);
    if (keff == 1) {
      if (c == 0) {
        if (tid < D) s_mean[tid] = (double)eth(0, tid);
        for (int i = tid; i < D * D; i += RT) {
          const int r = i / D, q = i % D;
          const double sd = 0.05 * ((double)a.hi[r] - (double)a.lo[r]);
          s_cov[i] = r == q ? sd * sd : 0.0;
        }
      }
    } else {
      // keff <= KSTAGE: the elites' values once into shared memory (X[d][e] as
      // FP64), centred after the mean, so that a covariance term is one FP64
      // multiply-add on shared operands; the sums run in the same order and
      // give the same values as the L2 path
      const bool staged = keff <= KSTAGE;
      const double invk = 1.0 / (double)keff;
      double* X = reinterpret_cast<double*>(dyn + sizeof(uint64_t) * (size_t)P);
      if (staged) {
        // two threads per elite, the loads of half a row in flight together
        constexpr int HALF = (CEM_MAX_D + 1) / 2;
        const int e = tid >> 1, d0 = (tid & 1) * HALF;
        if (e < keff) {
          const float* row = a.theta + (size_t)CEM_DIDX((int)(keys[e] & 0xFFFFF), a.N, 8) * D;
          float v[HALF];
#pragma unroll
          for (int q = 0; q < HALF; ++q) v[q] = d0 + q < D ? row[d0 + q] : 0.0f;
#pragma unroll
          for (int q = 0; q < HALF; ++q)
            if (d0 + q < D) X[(d0 + q) * keff + e] = (double)v[q];
        }
        static_assert(2 * KSTAGE <= RT, "two threads per staged elite");
        __syncthreads();
      }
      // a warp per output, lane l adding e = l, l + 32, ..., then a butterfly;
      // output o belongs to CTA o % nc
      for (int d = w * nc + c; d < D; d += 32 * nc) {
        double v = 0.0;
        if (staged)
          for (int e = lane; e < keff; e += 32) v += X[d * keff + e];
        else
          for (int e = lane; e < keff; e += 32) v += (double)eth(e, d);
        v = warp_sum(v);
        if (lane == 0) mean0[d] = v * invk;
      }
      sync_all();
      if (nc > 1 && c > 0 && tid < D) s_mean[tid] = mean0[tid];
      __syncthreads();
      if (staged) {
        for (int q = tid; q < keff * D; q += RT) X[q] -= s_mean[q / keff];
        __syncthreads();
      }
      const int npair = D * (D + 1) / 2;
      for (int p = w * nc + c; p < npair; p += 32 * nc) {
        int pj = p, pi = 0;  // pair index -> (pi, pj), pi <= pj
        while (pj >= D - pi) {
          pj -= D - pi;
          ++pi;
        }
        pj += pi;
        double v = 0.0;
        if (staged) {
          const double *xi = X + pi * keff, *xj = X + pj * keff;
          for (int e = lane; e < keff; e += 32) v += xi[e] * xj[e];
        } else {
          const double mi = s_mean[pi], mj = s_mean[pj];
          for (int e = lane; e < keff; e += 32) v += ((double)eth(e, pi) - mi) * ((double)eth(e, pj) - mj);
        }
        v = warp_sum(v);
        if (lane == 0) {
          double q = v * invk;
          if (pi == pj) {
            const double sd = 1e-4 * ((double)a.hi[pi] - (double)a.lo[pi]);
            q += sd * sd;
          }
          cov0[pi * D + pj] = q;
          cov0[pj * D + pi] = q;
        }
      }
    }
  }
  sync_all();
  if (c != 0) return;  // (nothing of the other CTAs' shared memory is read from here on)
  if (keff > 0) {
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
        const int b = CEM_DIDX((int)(keys[0] & 0xFFFFF), a.N, 8);
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
          for (int k = 0; k < 4; ++k) a.hist_cnt[4 * h + k] = total[k];
      }
      t->iter += 1;
    }
  }
}

__global__ void __launch_bounds__(RT) refit_kernel(RefitArgs a) { refit_body(a); }

// one cluster per problem of a batch; args[p] describes problem p
__global__ void __launch_bounds__(RT) refit_batch_kernel(const RefitArgs* __restrict__ args) {
  __shared__ RefitArgs a;
  const int nc = (int)cg::this_cluster().num_blocks();
  if (threadIdx.x == 0) a = args[blockIdx.x / nc];
  __syncthreads();
  if (a.skip) return;  // an eliminated plan keeps its state (all its CTAs leave)
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

static cudaError_t launch_clusters(const void* kernel, int clusters, int ctas, size_t smem, void** params,
                                   cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(clusters * ctas));
  cfg.blockDim = dim3(RT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, kernel, params);
}

cudaError_t launch_refit_batch(const RefitArgs* args_d, int n_problems, int maxN, int maxK, int maxD, cudaStream_t st) {
  if (n_problems <= 0) return cudaSuccess;
  void* params[] = {(void*)&args_d};
  return launch_clusters((const void*)refit_batch_kernel, n_problems, select_ctas(maxN), refit_smem_bytes(maxK, maxD),
                         params, st);
}

cudaError_t launch_refit(const RefitArgs& a, cudaStream_t st) {
  void* params[] = {(void*)&a};
  return launch_clusters((const void*)refit_kernel, 1, select_ctas(a.N), refit_smem_bytes(a.K, a.D), params, st);
}

}  // namespace cem
