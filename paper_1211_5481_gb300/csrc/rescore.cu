// rescore.cu -- candidate selection of the elite re-scoring: the n best
// chromosomes of a reduced-precision fitness vector, by (fitness, index) with
// NaN as +infinity (the ranking elitism uses, paper Section 3). Their fitness
// is then re-evaluated in FP64 by the Gram form (gram.cu) and replaces the
// reduced value, so elitism (Section 3; 2 elites, Section 5) and the
// tournaments rank the best candidates by accurate values.
//
// Two kernels. select_rank_kernel: a warp per chromosome counts, 32 at a time,
// the chromosomes that rank before it and gives up at n; the n that finish
// write their own place, and no CTA waits for another. Latency bound: one pass
// of the keys through shared memory, P / 32 ballots for the n best, a few for
// all others. (Selection and re-evaluation of 16 candidates, K = 257, P =
// 1024, with the re-evaluation's own change: 46 -> 16.9 us.) Above 16,384 chromosomes the launch of P
// warps and the long counts cost more than select_top_kernel (one CTA: each
// thread keeps the top 16 of its strided elements in registers, each warp
// merges its lanes' lists, warp 0 merges the 8 warps'). Fitness values are
// compared through order-preserving integer keys (integer compares instead of
// the FP64 pipe).
#include <math_constants.h>

#include "ga_device.cuh"
#include "game_internal.cuh"

namespace game {

namespace {

constexpr int kSelThreads = 256;

constexpr uint64_t kNoKey = ga::kKeyMax;

// Sorted list of kMaxRescore (key, index) pairs held in registers.
struct TopList {
  uint64_t k[kMaxRescore];
  int i[kMaxRescore];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int j = 0; j < kMaxRescore; ++j) {
      k[j] = kNoKey;
      i[j] = 0x7fffffff;
    }
  }
  __device__ __forceinline__ void insert(uint64_t key, int idx) {
    if (!ga::ranks_before(key, idx, k[kMaxRescore - 1], i[kMaxRescore - 1])) return;
    k[kMaxRescore - 1] = key;
    i[kMaxRescore - 1] = idx;
#pragma unroll
    for (int j = kMaxRescore - 1; j > 0; --j) {
      if (ga::ranks_before(k[j], i[j], k[j - 1], i[j - 1])) {
        const uint64_t tk = k[j];
        const int ti = i[j];
        k[j] = k[j - 1];
        i[j] = i[j - 1];
        k[j - 1] = tk;
        i[j - 1] = ti;
      }
    }
  }
  __device__ __forceinline__ void pop_front() {
#pragma unroll
    for (int j = 0; j < kMaxRescore - 1; ++j) {
      k[j] = k[j + 1];
      i[j] = i[j + 1];
    }
    k[kMaxRescore - 1] = kNoKey;
    i[kMaxRescore - 1] = 0x7fffffff;
  }
};

__global__ void __launch_bounds__(kSelThreads)
select_top_kernel(const double* __restrict__ fit, int P, int n, int* __restrict__ cand) {
  wait_previous();
  __shared__ uint64_t wk[kSelThreads / 32][kMaxRescore];
  __shared__ int wi[kSelThreads / 32][kMaxRescore];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  TopList L;
  L.clear();
  for (int p = tid; p < P; p += kSelThreads) L.insert(ga::rank_key(fit[p]), p);
  // each warp: n rounds of arg-min over its lanes' list heads
  for (int r = 0; r < n; ++r) {
    uint64_t k = L.k[0];
    int i = L.i[0];
    ga::warp_argmin(k, i);
    if (L.i[0] == i && i != 0x7fffffff) L.pop_front();
    if (lane == 0) {
      wk[warp][r] = k;
      wi[warp][r] = i;
    }
  }
  __syncthreads();
  if (warp != 0) return;
  L.clear();
#pragma unroll
  for (int j = 0; j < kMaxRescore; ++j)
    if (j < n && lane < kSelThreads / 32) {
      L.k[j] = wk[lane][j];
      L.i[j] = wi[lane][j];
    }
  for (int r = 0; r < n; ++r) {
    uint64_t k = L.k[0];
    int i = L.i[0];
    ga::warp_argmin(k, i);
    if (L.i[0] == i && i != 0x7fffffff) L.pop_front();
    if (lane == 0) cand[r] = i;
  }
}

constexpr int kRankMax = 16384;
constexpr int kRankWarps = 8;
constexpr int kRankChunk = 2048;   // keys staged in shared memory at a time
__global__ void __launch_bounds__(32 * kRankWarps)
select_rank_kernel(const double* __restrict__ fit, int P, int n, int* __restrict__ cand) {
  wait_previous();
  __shared__ uint64_t key[kRankChunk];
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * kRankWarps + (threadIdx.x >> 5);
  const uint64_t mine = i < P ? ga::rank_key(fit[i]) : kNoKey;
  int before = i < P ? 0 : n;
  for (int c0 = 0; c0 < P; c0 += kRankChunk) {
    const int len = min(kRankChunk, P - c0);
#pragma unroll 8
    for (int k = threadIdx.x; k < len; k += 32 * kRankWarps) key[k] = ga::rank_key(fit[c0 + k]);
    __syncthreads();
    for (int k0 = 0; k0 < len && before < n; k0 += 32) {
      const int k = k0 + lane;
      const bool b = k < len && ga::ranks_before(key[k], c0 + k, mine, i);
      before += __popc(__ballot_sync(0xffffffffu, b));
    }
    if (!__syncthreads_or(before < n)) break;
  }
  if (lane == 0 && before < n) cand[before] = i;
}

}  // namespace

cudaError_t launch_select_top(const double* fit, int P, int n, int* cand, bool callers,
                              cudaStream_t st) {
  if (n < 1) return cudaSuccess;
  if (n > kMaxRescore || n > P) return cudaErrorInvalidValue;
  const int grid = P <= kRankMax ? ceil_div(P, kRankWarps) : 1;
  const auto kern = P <= kRankMax ? select_rank_kernel : select_top_kernel;
  constexpr int threads = 32 * kRankWarps;
  static_assert(threads == kSelThreads, "both selections");
  // The fitness is read through L1 (past it, P = 16,384 takes 82 us for 60), so behind
  // a caller's kernel, which may release its successor while it still writes, the
  // launch is an ordinary one.
  if (callers) {
    kern<<<grid, threads, 0, st>>>(fit, P, n, cand);
    return cudaGetLastError();
  }
  return launch_behind(kern, grid, threads, 0, st, fit, P, n, cand);
}

}  // namespace game
