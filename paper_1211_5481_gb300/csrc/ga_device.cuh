// ga_device.cuh -- the GA operators as device functions, shared by the
// single-problem kernels (ga_ops.cu) and the batched ones (batch.cu). The
// definitions (ranking key, parent selection, crossover, mutation,
// immigrants) are documented in ga_ops.cu.
#pragma once
#include <math_constants.h>

#include "game_internal.cuh"
#include "philox.cuh"

namespace game {
namespace ga {

constexpr int kPlanThreads = 1024;
constexpr int kMaxElites = 256;

// Ranking key of a fitness value as an unsigned integer whose order is the
// order of the values (NaN as +infinity, -0 as +0, so equal values tie as in
// FP64 comparison): the GPU ranks with integer compares instead of the slow
// FP64 pipe.
__device__ __forceinline__ uint64_t rank_key(double f) {
  constexpr uint64_t kInf = 0x7ff0000000000000ull, kSign = 0x8000000000000000ull;
  const uint64_t u = (uint64_t)__double_as_longlong(f);
  if ((u & ~kSign) > kInf) return kInf | kSign;   // NaN
  return (u >> 63) && u != kSign ? ~u : (u | kSign);
}
constexpr uint64_t kKeyMax = ~0ull;   // above every rank_key

// (ka, a) ranks before (kb, b)
__device__ __forceinline__ bool ranks_before(uint64_t ka, int a, uint64_t kb, int b) {
  return ka < kb || (ka == kb && a < b);
}

// Warp-wide arg-min by (key, index); every lane receives the winner. Three
// 32-bit reductions instead of five shuffle rounds of a 64-bit key and an index.
__device__ __forceinline__ void warp_argmin(uint64_t& k, int& i) {
  const uint32_t hi = (uint32_t)(k >> 32), lo = (uint32_t)k;
  const uint32_t mh = __reduce_min_sync(0xffffffffu, hi);
  const uint32_t ml = __reduce_min_sync(0xffffffffu, hi == mh ? lo : 0xffffffffu);
  const bool win = hi == mh && lo == ml;
  i = (int)__reduce_min_sync(0xffffffffu, win ? (uint32_t)i : 0x7fffffffu);
  k = ((uint64_t)mh << 32) | ml;
}

// Gene e = p K + k of the initial population (uniform in [-1, 1)).
__device__ __forceinline__ float init_gene(uint64_t seed, int K, int64_t e) {
  const uint32_t p = (uint32_t)(e / K), k = (uint32_t)(e % K);
  return uniform_gene(philox4x32_10(seed, 0u, p, k, kTagInit).x);
}

// Roulette weight of a fitness value: floor(2^32 RN(1 / RN(1 + f))), 0 for
// a NaN, negative or infinite f (all operations IEEE round-to-nearest).
__device__ __forceinline__ uint64_t roulette_weight(double f) {
  if (!(f >= 0.0) || isinf(f)) return 0;
  const double w = __ddiv_rn(1.0, __dadd_rn(1.0, f));
  return __double2ull_rz(__dmul_rn(w, 4294967296.0));
}

// Parent r (0 or 1) of pair q, drawn from the ga.P current chromosomes.
// Every mode takes its words from Philox(seed; g, q, r, TOUR | call << 8).
__device__ __forceinline__ int select_parent(const GaDev& ga, const double* __restrict__ fit,
                                             uint64_t seed, uint32_t g, uint32_t q, uint32_t r) {
  if (ga.sel == GAME_SEL_RANKING) {
    // u uniform on [0, P (P + 1) / 2); rank k covers C(k) <= u < C(k + 1),
    // C(k) = sum_{j<k} (P - j) = k P - k (k - 1) / 2
    const uint32_t x = philox4x32_10(seed, g, q, r, kTagTour).x;
    const uint64_t P = (uint64_t)ga.P;
    const uint64_t u = ((uint64_t)x * (P * (P + 1) / 2)) >> 32;
    int lo = 0, hi = ga.P - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      const uint64_t c = (uint64_t)mid * P - (uint64_t)mid * (uint64_t)(mid - 1) / 2;
      if (c <= u) lo = mid;
      else hi = mid - 1;
    }
    return ga.order[lo];
  }
  if (ga.sel == GAME_SEL_ROULETTE) {
    // u uniform on [0, W) from 64 bits; chromosome p covers [cum[p], cum[p + 1])
    const uint4 w = philox4x32_10(seed, g, q, r, kTagTour);
    const uint64_t W = ga.cum[ga.P];
    if (W == 0) return (int)(((uint64_t)w.x * (uint64_t)ga.P) >> 32);
    const uint64_t u = __umul64hi(((uint64_t)w.x << 32) | w.y, W);
    int lo = 0, hi = ga.P - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (u < ga.cum[mid + 1]) hi = mid;
      else lo = mid + 1;
    }
    return lo;
  }
  // tournament: the best of T uniform candidates
  int win = -1;
  uint64_t wk = 0;
  uint4 w = make_uint4(0, 0, 0, 0);
  for (int s = 0; s < ga.T; ++s) {
    if ((s & 3) == 0) w = philox4x32_10(seed, g, q, r, kTagTour | ((uint32_t)(s >> 2) << 8));
    const uint32_t word = (s & 3) == 0 ? w.x : (s & 3) == 1 ? w.y : (s & 3) == 2 ? w.z : w.w;
    const int c = (int)(((uint64_t)word * (uint64_t)ga.P) >> 32);
    const uint64_t ck = rank_key(fit[c]);
    if (win < 0 || ranks_before(ck, c, wk, win)) {
      win = c;
      wk = ck;
    }
  }
  return win;
}

__host__ __device__ inline int pow2_at_least(int P) {
  int n2 = 1;
  while (n2 < P) n2 <<= 1;
  return n2;
}

// Ranks by counting, for populations up to kCountMax: thread groups of T share a
// chromosome, each thread compares it with every T-th other, so a rank takes
// P / T compares and a few shuffles. put(rank, chromosome) once per chromosome.
// A bitonic sort of 32 keys by the same 1024 threads took 11,200 cycles (a
// block barrier per step), an arg-min per elite 2,700; this 400. Beyond 512
// the P^2 compares cost more than the sort. key [P] in shared memory.
constexpr int kCountMax = 512;
template <class Put>
__device__ __forceinline__ void count_ranks(int P, const double* __restrict__ fit, uint64_t* key,
                                            Put put) {
  int T = kPlanThreads / 32;   // threads per chromosome
  while (T > 1 && T * P > kPlanThreads) T >>= 1;
  for (int i = threadIdx.x; i < P; i += kPlanThreads) key[i] = rank_key(fit[i]);
  __syncthreads();
  const int i = threadIdx.x / T, sub = threadIdx.x % T;
  int c = 0;
  if (i < P) {
    const uint64_t k = key[i];
    for (int j = sub; j < P; j += T) c += ranks_before(key[j], j, k, i) ? 1 : 0;
  }
  for (int o = T >> 1; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (i < P && sub == 0) put(c, i);
  __syncthreads();
}

// order[r] = the chromosome of rank r (order may be NULL: the result stays in
// sidx): a bitonic sort of (rank key, index) over the next power of two
// >= P, padded with keys above every chromosome; skey [n2] and sidx [n2] in
// shared memory.
__device__ __forceinline__ void ranking_sort_body(int P, const double* __restrict__ fit, uint64_t* skey,
                                  int* sidx, int* __restrict__ order) {
  if (P <= kCountMax) {
    count_ranks(P, fit, skey, [&](int r, int i) {
      sidx[r] = i;
      if (order) order[r] = i;
    });
    return;
  }
  const int n2 = pow2_at_least(P);
  for (int i = threadIdx.x; i < n2; i += kPlanThreads) {
    skey[i] = i < P ? ga::rank_key(fit[i]) : ga::kKeyMax;
    sidx[i] = i < P ? i : 0x7fffffff;
  }
  __syncthreads();
  for (int k = 2; k <= n2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < n2; i += kPlanThreads) {
        const int l = i ^ j;
        if (l <= i) continue;
        const bool up = (i & k) == 0;   // ascending run
        const bool swap = up ? ga::ranks_before(skey[l], sidx[l], skey[i], sidx[i])
                             : ga::ranks_before(skey[i], sidx[i], skey[l], sidx[l]);
        if (swap) {
          const uint64_t tk = skey[i];
          skey[i] = skey[l];
          skey[l] = tk;
          const int ti = sidx[i];
          sidx[i] = sidx[l];
          sidx[l] = ti;
        }
      }
      __syncthreads();
    }
  if (order)
    for (int i = threadIdx.x; i < P; i += kPlanThreads) order[i] = sidx[i];
}

// cum[p + 1] = sum_{j<=p} roulette_weight(fit[j]), cum[0] = 0: each thread
// sums a contiguous chunk, an exclusive scan of the chunk sums gives its
// offset (integers, so the result does not depend on the order).
__device__ __forceinline__ void roulette_cum_body(int P, const double* __restrict__ fit, uint64_t* cum) {
  __shared__ uint64_t wsum[kPlanThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int chunk = (P + kPlanThreads - 1) / kPlanThreads;
  const int lo = min(P, tid * chunk), hi = min(P, lo + chunk);
  uint64_t s = 0;
  for (int p = lo; p < hi; ++p) s += ga::roulette_weight(fit[p]);
  uint64_t inc = s;   // inclusive scan within the warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) wsum[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    uint64_t t = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t v = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += v;
    }
    wsum[lane] = t;   // inclusive over warps
  }
  __syncthreads();
  uint64_t run = (wid > 0 ? wsum[wid - 1] : 0) + inc - s;
  for (int p = lo; p < hi; ++p) {
    run += ga::roulette_weight(fit[p]);
    cum[p + 1] = run;
  }
  if (tid == 0) cum[0] = 0;
}

// bytes of the selection table when it is kept in shared memory
__host__ __device__ inline int table_bytes(const GaDev& ga) {
  return ga.sel == GAME_SEL_RANKING    ? pow2_at_least(ga.P) * 12
         : ga.sel == GAME_SEL_ROULETTE ? (ga.P + 1) * 8
                                       : 0;
}

// CTA `block` of `blocks`, kPlanThreads threads: elites (the first CTA), parent selection and crossover plan of
// one problem (plan[s] = {head parent, tail parent, cut, elite flag}) for
// ga.Nout output slots; tournaments draw from the ga.P current chromosomes.
__device__ __forceinline__ void plan_body(const GaDev& ga, const double* __restrict__ fit,
                                          uint64_t seed, uint32_t g, int4* __restrict__ plan,
                                          int block = 0, int blocks = 1) {
  __shared__ int elite[kMaxElites];
  __shared__ uint64_t wkey[kPlanThreads / 32];
  __shared__ int widx[kPlanThreads / 32];
  __shared__ uint64_t key[kCountMax];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // 1. elites: the first ranks where the selection sorted the population, else by
  // counting (P^2 compares, whatever the number of elites) or by one block-wide
  // arg-min per elite. us per generation of a tiny run (M = 100, K = 3), counting /
  // arg-min: P = 72: 12.2 / 12.0 (1 elite), 12.0 / 12.3 (2); 128: 13.1 / 12.9 (2);
  // 200: 15.7 / 15.1 (4); 256: 16.9 / 17.3 (8); 300: 18.7 / 17.8 (8); 400: 23.0 /
  // 23.7 (16); 512: 27.5 / 15.8 (2), 27.4 / 36.6 (32).
  if (block != 0) {
  } else if (ga.sel == GAME_SEL_RANKING) {
    for (int e = tid; e < ga.E; e += kPlanThreads) elite[e] = ga.order[e];
    __syncthreads();
  } else if (ga.P <= kCountMax && ga.P * ga.P <= 8000 * ga.E) {
    count_ranks(ga.P, fit, key, [&](int r, int i) {
      if (r < ga.E) elite[r] = i;
    });
  } else {
    for (int e = 0; e < ga.E; ++e) {
      uint64_t bk = kKeyMax;
      int bi = 0x7fffffff;
      for (int p = tid; p < ga.P; p += kPlanThreads) {
        bool taken = false;
        for (int j = 0; j < e; ++j) taken |= (elite[j] == p);
        if (taken) continue;
        const uint64_t k = rank_key(fit[p]);
        if (ranks_before(k, p, bk, bi)) {
          bk = k;
          bi = p;
        }
      }
      warp_argmin(bk, bi);
      if (lane == 0) {
        wkey[wid] = bk;
        widx[wid] = bi;
      }
      __syncthreads();
      if (wid == 0) {
        bk = wkey[lane];
        bi = widx[lane];
        warp_argmin(bk, bi);
        if (lane == 0) elite[e] = bi;
      }
      __syncthreads();
    }
  }
  if (block == 0)
    for (int e = tid; e < ga.E; e += kPlanThreads)
      plan[e] = make_int4(elite[e], elite[e], ga.K, 1);

  // 2.-3. pairs: the two parents and the crossover decision, a thread each
  const int npairs = (ga.Nout - ga.E + 1) / 2;
  int* words = reinterpret_cast<int*>(plan);
  for (int t = block * kPlanThreads + tid; t < 3 * npairs; t += blocks * kPlanThreads) {
    const int q = t / 3, r = t - 3 * q;
    const int s0 = ga.E + 2 * q;
    int* w0 = words + 4 * (int64_t)s0;   // slot s0's {head, tail, cut, elite}
    const bool two = s0 + 1 < ga.Nout;
    if (r < 2) {
      const int parent = select_parent(ga, fit, seed, g, (uint32_t)q, (uint32_t)r);
      w0[r] = parent;
      if (two) w0[4 + (r ^ 1)] = parent;
    } else {
      const uint4 wx = philox4x32_10(seed, g, (uint32_t)q, 0u, kTagCross);
      int cut = ga.K;
      if ((wx.x >> 8) < ga.thr_pc)
        cut = 1 + (int)(((uint64_t)wx.y * (uint64_t)(ga.K - 1)) >> 32);
      w0[2] = cut;
      w0[3] = 0;
      if (two) {
        w0[6] = cut;
        w0[7] = 0;
      }
    }
  }
}

// Gene e = s K + k of the next population.
__device__ __forceinline__ float breed_gene(const GaDev& ga, const float* __restrict__ pop,
                                            const int4* __restrict__ plan, uint64_t seed,
                                            uint32_t g, int64_t e) {
  int s, k;   // 32-bit division where it does
  if ((uint64_t)e < 0x80000000ull) {
    s = (int)((uint32_t)e / (uint32_t)ga.K);
    k = (int)((uint32_t)e - (uint32_t)s * (uint32_t)ga.K);
  } else {
    s = (int)(e / ga.K);
    k = (int)(e % ga.K);
  }
  float v;
  if (s >= ga.Nout - ga.I) {
    v = uniform_gene(philox4x32_10(seed, g, (uint32_t)s, (uint32_t)k, kTagImmigrant).x);
  } else {
    const int4 pl = plan[s];
    v = pop[(int64_t)(k < pl.z ? pl.x : pl.y) * ga.K + k];
    if (s >= ga.E) {
      const uint4 w = philox4x32_10(seed, g, (uint32_t)s, (uint32_t)k, kTagMut);
      if ((w.x >> 8) < ga.thr_pm) {
        const float z = irwin_hall12(seed, g, (uint32_t)s, (uint32_t)k);
        v = __fadd_rn(v, __fmul_rn(ga.sigma, z));
        if (v < -1.0f) v = -1.0f;
        if (v > 1.0f) v = 1.0f;
      }
    }
  }
  return v;
}

}  // namespace ga
}  // namespace game
