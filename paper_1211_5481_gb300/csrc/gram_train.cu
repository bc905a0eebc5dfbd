// gram_train.cu -- whole generations of a small Gram-form run in one launch.
//
// What bounded such runs (the paper's experiment: 19 chromosomes of 17 shared
// genes): two dependent launches a generation whose work is a few thousand
// FP64 operations, 29 us a generation with the stop rule's read-back. Here a
// cluster of 8 CTAs keeps the population, the fitness, the Gram form's pair
// list and the plan in shared memory and runs up to thousands of generations:
// every CTA plans and breeds the whole population (the operators are counter-
// based, so all get the same), evaluates every 8th chromosome and writes its
// fitness into all 8 shared memories; one cluster barrier ends the generation.
// The stop rule runs on the device. Operators and fitness are those of the
// separate kernels bit for bit (ga_device.cuh, quad_pairs).
// Measured: the paper's set (M = 2100, trigonometric degree 8, shared genes,
// ranking, P = 19, stop rule every 10 generations): 5.7 us a
// generation.
#include "ga_device.cuh"
#include "fp64.cuh"
#include "game_internal.cuh"
#include "gram.cuh"
#include "tc_ptx.cuh"

namespace game {

namespace {

constexpr int kCluster = 8;
constexpr int kWarps = ga::kPlanThreads / 32;
// Every CTA plans and breeds the whole population, so beyond 96 chromosomes the
// separate kernels are faster. us for 20 generations, separate kernels / one
// launch, tournament, K = 5: P = 19: 147 / 108; 64: 159 / 134; 96: 168 / 167; 128:
// 181 / 194; 300: 279 / 443; 1000: 329 / 896; K = 17, P = 96: 209 / 215, ranking
// 220 / 216. (One generation alone pays the set-up: 16.3 / 18.9 at P = 19, 17.2 /
// 22.1 at P = 96.)
constexpr int kMaxP = 96;
constexpr int kMaxSmem = 200 * 1024;
// FP64 operations of one CTA's chromosomes per generation above which the
// separate kernels, with the whole GPU's FP64 pipes, are faster: one SM does
// two a cycle, so 24,000 take about 6 us, what the two launches cost.
constexpr int64_t kMaxOps = 24000;

struct Layout {
  int Gp, b, fit, row, table, plan, pop, kk, total;
};

__host__ __device__ inline Layout layout(const GaDev& g) {
  const int E = g.K * (g.K + 1) / 2;
  Layout l;
  l.Gp = 0;
  l.b = l.Gp + 8 * E;
  l.fit = l.b + 8 * g.K;
  l.row = l.fit + 16 * g.P;
  l.table = (l.row + kWarps * kPairK * 8 + 15) & ~15;
  l.plan = l.table + ((ga::table_bytes(g) + 15) & ~15);
  l.pop = l.plan + 16 * g.P;
  l.kk = l.pop + 8 * g.P * g.K;
  l.total = l.kk + 2 * E;
  return l;
}

struct TrainArgs {
  GaDev ga;
  int err, gens, done0, every;   // every: 0, or generations between stop checks
  int64_t M;
  double threshold;
  uint64_t seed;
  uint32_t g0;
  const float* pop_in;
  float* pop_out;
  double* fit;
  const double *Gp, *b, *yy;
  const uint16_t* kk;
  int* done;   // generations run
};

__global__ void __launch_bounds__(ga::kPlanThreads) gram_train_kernel(const TrainArgs a) {
  extern __shared__ __align__(16) uint8_t smem[];
  GaDev ga = a.ga;
  const int P = ga.P, K = ga.K, E = K * (K + 1) / 2;
  const Layout l = layout(ga);
  double* Gp = reinterpret_cast<double*>(smem + l.Gp);
  double* b = reinterpret_cast<double*>(smem + l.b);
  double* fit = reinterpret_cast<double*>(smem + l.fit);      // [2][P]
  uint64_t* table = reinterpret_cast<uint64_t*>(smem + l.table);
  int4* plan = reinterpret_cast<int4*>(smem + l.plan);
  float* pop = reinterpret_cast<float*>(smem + l.pop);        // [2][P K]
  uint16_t* kk = reinterpret_cast<uint16_t*>(smem + l.kk);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* row = reinterpret_cast<double*>(smem + l.row) + warp * kPairK;
  const uint32_t rank = ptx::cluster_ctarank();
  for (int e = tid; e < E; e += ga::kPlanThreads) {
    Gp[e] = a.Gp[e];
    kk[e] = a.kk[e];
  }
  for (int k = tid; k < K; k += ga::kPlanThreads) b[k] = a.b[k];
  for (int p = tid; p < P; p += ga::kPlanThreads) fit[p] = a.fit[p];
  for (int e = tid; e < P * K; e += ga::kPlanThreads) pop[e] = a.pop_in[e];
  const double yy = *a.yy, dM = (double)a.M, rM = 1.0 / dM;
  __syncthreads();
  ptx::cluster_sync();   // every CTA runs before anyone writes to it

  int cur = 0, n = 0;
  for (; n < a.gens; ++n) {
    const double* f = fit + cur * P;
    if (a.every > 0 && (a.done0 + n) % a.every == 0) {
      if (__syncthreads_or(tid < P && f[tid] < a.threshold)) break;   // the same in every CTA
    }
    if (ga.sel == GAME_SEL_RANKING) {
      int* order = reinterpret_cast<int*>(table + ga::pow2_at_least(P));
      ga::ranking_sort_body(P, f, table, order, nullptr);
      ga.order = order;
    } else if (ga.sel == GAME_SEL_ROULETTE) {
      ga::roulette_cum_body(P, f, table);
      ga.cum = table;
    }
    __syncthreads();
    const uint32_t g = a.g0 + (uint32_t)n;
    ga::plan_body(ga, f, a.seed, g, plan);
    __syncthreads();
    const float* from = pop + cur * P * K;
    float* next = pop + (cur ^ 1) * P * K;
    for (int e = tid; e < P * K; e += ga::kPlanThreads)
      next[e] = ga::breed_gene(ga, from, plan, a.seed, g, e);
    __syncthreads();
    double* fn = fit + (cur ^ 1) * P;
    for (int p = (int)rank + kCluster * warp; p < P; p += kCluster * kWarps) {
      for (int k = lane; k < K; k += 32) row[k] = (double)next[p * K + k];
      __syncwarp();
      const double v = finish_error(divide_by(yy + quad_pairs(K, row, Gp, kk, b, lane), dM, rM), a.err);
      if (lane < kCluster)
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(
                         ptx::mapa(ptx::smem_addr(fn + p), (uint32_t)lane)),
                     "d"(v)
                     : "memory");
      __syncwarp();
    }
    ptx::cluster_sync();
    cur ^= 1;
  }
  if (rank == 0) {
    if (n > 0) {
      for (int e = tid; e < P * K; e += ga::kPlanThreads) a.pop_out[e] = pop[cur * P * K + e];
      for (int p = tid; p < P; p += ga::kPlanThreads) a.fit[p] = fit[cur * P + p];
    }
    if (tid == 0) *a.done = n;
  }
}

}  // namespace

bool gram_train_fits(const GaDev& g) {
  if (g.K > kPairK || g.P > kMaxP || g.E > ga::kMaxElites || g.Nout != g.P) return false;
  const int64_t E = (int64_t)g.K * (g.K + 1) / 2;
  return 2 * E * ceil_div(g.P, kCluster) <= kMaxOps && layout(g).total <= kMaxSmem;
}

cudaError_t launch_gram_train(const GaDev& g, const GramDev& gram, int64_t M, int err,
                              const float* pop_in, float* pop_out, double* fit, uint64_t seed,
                              uint32_t g0, int gens, int done0, int every, double threshold,
                              int* done, cudaStream_t st) {
  if (!gram_train_fits(g) || gens < 1) return cudaErrorInvalidValue;
  TrainArgs a;
  a.ga = g;
  a.err = err;
  a.gens = gens;
  a.done0 = done0;
  a.every = every;
  a.M = M;
  a.threshold = threshold;
  a.seed = seed;
  a.g0 = g0;
  a.pop_in = pop_in;
  a.pop_out = pop_out;
  a.fit = fit;
  a.Gp = gram.list;
  a.b = gram.b;
  a.yy = gram.yy;
  a.kk = gram.kk;
  a.done = done;
  cudaError_t e = cudaFuncSetAttribute(gram_train_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCluster);
  cfg.blockDim = dim3(ga::kPlanThreads);
  cfg.dynamicSmemBytes = (size_t)layout(g).total;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, gram_train_kernel, a);
}

}  // namespace game
