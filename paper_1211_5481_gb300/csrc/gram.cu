// gram.cu -- the Gram form of the MSE fitness (FP64).
//
// With phi~(x) = (1, phi_1(x), ..., phi_{K-1}(x)) the expansion of Eq. 1 /
// Eq. 6 with a leading 1 for the bias gene, the output of Eq. 2 is
// Out_p(m) = a_p . phi~(x_m), so the MSE of Eq. 3 is a quadratic form:
//   fit_p = (yy - 2 a_p . b + a_p^T G a_p) / M,
//   G = sum_m phi~(x_m) phi~(x_m)^T [K][K], b = sum_m y_m phi~(x_m), yy = sum_m y_m^2.
// G, b and yy depend only on the training set: they are accumulated once per
// handle (FP64 expansion -- the Chebyshev recurrence, or sin / cos of x and
// the angle recurrence -- and FP64 sums), after which a generation costs
// P K^2 FP64 multiply-adds instead of M P K. The subtraction cancels when the
// fit is good (fit << yy / M), which is why everything here is FP64.
//
// Shared genes (Eq. 2 as printed): the expansion is
// psi~(x) = (1, psi_1(x), ..., psi_{B d}(x)) with psi_{b,j}(x) =
// sum_i phi_{b,j}(x_i) (features in order), written by expand_tied_kernel;
// everything else is the same with K = B d + 1.
// The MSE is clamped at 0 against cancellation; RMSE is its square root.
//
// Accumulation: the patterns are taken in chunks of up to kChunk; a chunk's
// design matrix Phi [mc][K] (FP64) is written by expand_kernel, then
// gram_accum_kernel forms Phi^T Phi on the upper triangle (64 x 64 tiles,
// each thread a 4 x 4 block) over up to 32 row ranges of the chunk, each in
// row order, and gram_add_kernel adds the ranges' sums to G in range order;
// vec_accum_kernel / vec_add_kernel do the same for Phi^T y and y^T y over 64
// row ranges. Every sum runs in a fixed order (chunks in sequence, ranges
// in order, rows in order within a range), so G is reproducible.
// The quadratic forms use G's symmetry, so a chromosome costs about K^2 / 2
// FP64 multiply-adds (an SM issues two a cycle: the FP64 pipe bounds all of
// this); quad_rows_kernel and quad_pairs_kernel (gram.cuh) below.
#include <math_constants.h>

#include "game_internal.cuh"
#include "gram.cuh"

namespace game {

namespace {

constexpr int kGT = 64;        // G tile
constexpr int kVecSplits = 64; // row splits of a chunk's b and y.y sums

// Phi[r][k] for patterns m0 + r (r < mc), FP64; column 0 is 1.
__global__ void expand_kernel(int64_t m0, int mc, int N, int d, int basis, int K,
                              const float* __restrict__ Xt, double* __restrict__ Phi) {
  const int B = basis == GAME_BASIS_TRIG ? 2 : 1;
  const int64_t n = (int64_t)mc * N;   // one thread per (pattern, feature)
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(e / N), i = (int)(e % N);
    const int64_t m = m0 + r;
    const double x =
        (double)Xt[(m / kPatBlock) * (int64_t)N * kPatBlock + (int64_t)i * kPatBlock + m % kPatBlock];
    double* row = Phi + (int64_t)r * K;
    if (i == 0) row[0] = 1.0;
    const int64_t base = 1 + (int64_t)i * B * d;
    if (basis == GAME_BASIS_CHEB) {
      double tm = 1.0, t = x;
      for (int j = 1; j <= d; ++j) {
        row[base + j - 1] = t;
        const double tn = 2.0 * x * t - tm;
        tm = t;
        t = tn;
      }
    } else {
      double s1, c1;
      sincos(x, &s1, &c1);
      for (int bb = 0; bb < 2; ++bb) {
        double fm = bb ? 0.0 : 1.0, f = bb ? s1 : c1;
        for (int j = 1; j <= d; ++j) {
          row[base + bb * d + j - 1] = f;
          const double fn = 2.0 * c1 * f - fm;
          fm = f;
          f = fn;
        }
      }
    }
  }
}

// Psi[r][c] for patterns m0 + r with shared genes: column 0 is 1, column
// 1 + b d + (j - 1) the sum over features i = 0..N-1, in order, of
// phi_{b,j}(x_i); K = B d + 1.
__global__ void expand_tied_kernel(int64_t m0, int mc, int N, int d, int basis, int K,
                                   const float* __restrict__ Xt, double* __restrict__ Phi) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < mc; r += gridDim.x * blockDim.x) {
    const int64_t m = m0 + r;
    double* row = Phi + (int64_t)r * K;
    row[0] = 1.0;
    for (int c = 1; c < K; ++c) row[c] = 0.0;
    for (int i = 0; i < N; ++i) {
      const double x = (double)Xt[(m / kPatBlock) * (int64_t)N * kPatBlock +
                                  (int64_t)i * kPatBlock + m % kPatBlock];
      if (basis == GAME_BASIS_CHEB) {
        double tm = 1.0, t = x;
        for (int j = 1; j <= d; ++j) {
          row[j] += t;
          const double tn = 2.0 * x * t - tm;
          tm = t;
          t = tn;
        }
      } else {
        double s1, c1;
        sincos(x, &s1, &c1);
        for (int bb = 0; bb < 2; ++bb) {
          double fm = bb ? 0.0 : 1.0, f = bb ? s1 : c1;
          for (int j = 1; j <= d; ++j) {
            row[1 + bb * d + j - 1] += f;
            const double fn = 2.0 * c1 * f - fm;
            fm = f;
            f = fn;
          }
        }
      }
    }
  }
}

// part[z][k1][k2] = sum over rows r of split z of Phi[r][k1] Phi[r][k2], for
// the tile (blockIdx.y, blockIdx.x) of the upper triangle (tiles with
// ti > tj skip); split z = blockIdx.z takes rows [z rs, (z + 1) rs).
__global__ void __launch_bounds__(256)
gram_accum_kernel(int mc, int rs, int K, const double* __restrict__ Phi,
                  double* __restrict__ part) {
  const int ti = blockIdx.y, tj = blockIdx.x;
  if (ti > tj) return;
  const int rlo = blockIdx.z * rs, rhi = min(mc, rlo + rs);
  __shared__ double Ps[16][2 * kGT];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int k10 = ti * kGT, k20 = tj * kGT;
  double acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0.0;
  for (int r0 = rlo; r0 < rhi; r0 += 16) {
    for (int e = threadIdx.x; e < 16 * 2 * kGT; e += 256) {
      const int rr = e / (2 * kGT), c = e % (2 * kGT);
      const int k = c < kGT ? k10 + c : k20 + (c - kGT);
      Ps[rr][c] = (r0 + rr < rhi && k < K) ? Phi[(int64_t)(r0 + rr) * K + k] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int rr = 0; rr < 16; ++rr) {
      double a[4], bv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) a[u] = Ps[rr][ty + 16 * u];
#pragma unroll
      for (int v = 0; v < 4; ++v) bv[v] = Ps[rr][kGT + tx + 16 * v];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = fma(a[u], bv[v], acc[u][v]);
    }
    __syncthreads();
  }
  double* Pz = part + (int64_t)blockIdx.z * K * K;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int k1 = k10 + ty + 16 * u, k2 = k20 + tx + 16 * v;
      if (k1 < K && k2 < K && k1 <= k2) Pz[(int64_t)k1 * K + k2] = acc[u][v];
    }
}

// G[k1][k2] += sum over the splits, in order, of part[z][k1][k2] (upper triangle).
__global__ void gram_add_kernel(int K, int splits, const double* __restrict__ part,
                                double* __restrict__ G) {
  const int64_t n = (int64_t)K * K;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int k1 = (int)(e / K), k2 = (int)(e % K);
    if (k1 > k2) continue;
    double s = 0.0;
    for (int z = 0; z < splits; ++z) s += part[z * n + e];
    G[e] += s;
  }
}

// vpart[z][k] = sum over the rows r of split z (in order) of Phi[r][k] y[m0 + r]
// for k < K, and vpart[z][K] = sum of y[m0 + r]^2; split z = blockIdx.y
// takes rows [z rs, (z + 1) rs). Threads of a block read consecutive
// columns of a row (coalesced).
__global__ void vec_accum_kernel(int64_t m0, int mc, int rs, int K, const double* __restrict__ Phi,
                                 const float* __restrict__ y, double* __restrict__ vpart) {
  const int rlo = blockIdx.y * rs, rhi = min(mc, rlo + rs);
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= K; k += gridDim.x * blockDim.x) {
    double s = 0.0;
    if (k < K) {
      for (int r = rlo; r < rhi; ++r) s = fma(Phi[(int64_t)r * K + k], (double)y[m0 + r], s);
    } else {
      for (int r = rlo; r < rhi; ++r) {
        const double v = y[m0 + r];
        s = fma(v, v, s);
      }
    }
    vpart[(int64_t)blockIdx.y * (K + 1) + k] = s;
  }
}

// b[k] += sum over the splits, in order, of vpart[z][k]; yy likewise from column K.
__global__ void vec_add_kernel(int K, int splits, const double* __restrict__ vpart,
                               double* __restrict__ b, double* __restrict__ yy) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k > K) return;
  double s = 0.0;
  for (int z = 0; z < splits; ++z) s += vpart[(int64_t)z * (K + 1) + k];
  if (k < K) b[k] += s;
  else *yy += s;
}

// Lower triangle from the upper one.
__global__ void mirror_kernel(int K, double* __restrict__ G) {
  const int64_t n = (int64_t)K * K;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int k1 = (int)(e / K), k2 = (int)(e % K);
    if (k1 > k2) G[e] = G[(int64_t)k2 * K + k1];
  }
}

// Pair list of a small form (K <= kPairK): entry e < K (K + 1) / 2 is the pair
// k1 <= k2 in row order, with weight G[k1][k1] or 2 G[k1][k2].
__global__ void pairs_kernel(int K, const double* __restrict__ G, double* __restrict__ Gp,
                             uint16_t* __restrict__ kk) {
  for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
    const int k1 = e / K, k2 = e % K;
    if (k1 > k2) continue;
    const int at = k1 * K - k1 * (k1 - 1) / 2 + (k2 - k1);
    Gp[at] = k1 == k2 ? G[e] : 2.0 * G[e];
    kk[at] = (uint16_t)(k1 | (k2 << 8));
  }
}

// K <= kPairK: one warp per chromosome (quad_pairs in gram.cuh).
constexpr int kPairWarps = 4;
__global__ void __launch_bounds__(32 * kPairWarps)
quad_pairs_kernel(int P, int K, double m, double rm, int err, const float* __restrict__ pop,
                  const int* __restrict__ idx, const double* __restrict__ Gp,
                  const uint16_t* __restrict__ kk, const double* __restrict__ b,
                  const double* __restrict__ yy, double* __restrict__ fit) {
  wait_previous();
  __shared__ double as[kPairWarps][kPairK];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int q = blockIdx.x * kPairWarps + warp;
  if (q >= P) return;
  const int p = idx ? idx[q] : q;
  for (int k = lane; k < K; k += 32) as[warp][k] = (double)__ldcg(pop + (int64_t)p * K + k);
  __syncwarp();
  const double v = quad_pairs(K, as[warp], Gp, kk, b, lane);
  if (lane == 0) fit[p] = finish_error(divide_by(*yy + v, m, rm), err);
}

// Larger K. Rows are taken in blocks of 32 (lane = row); block I needs the
// columns k2 >= 32 I only: its own 32 x 32 square once, everything to the right
// twice. The (block, column) steps of all blocks form one list, laid out once
// per handle (steps_kernel: a step's 32 weighted entries of G side by side).
constexpr int kAheadMax = 20;     // steps a warp loads ahead (the list is padded by them)
__host__ __device__ inline int64_t row_steps(int K) {
  const int64_t NB = (K + 31) / 32;
  return NB * K - 16 * NB * (NB - 1);   // sum over I of (K - 32 I)
}
__global__ void steps_kernel(int K, const double* __restrict__ G, double* __restrict__ T) {
  const int I = blockIdx.x, lane = threadIdx.x & 31;
  const int64_t base = (int64_t)I * K - 16ll * I * (I - 1);
  const int k1 = 32 * I + lane;
  for (int c = blockIdx.y * 8 + (threadIdx.x >> 5); c < K - 32 * I; c += gridDim.y * 8) {
    const double g = k1 < K ? G[(int64_t)(32 * I + c) * K + k1] : 0.0;
    T[(base + c) * 32 + lane] = c < 32 ? g : 2.0 * g;
  }
}

// The list is cut into kQuadRanges contiguous ranges; a warp takes a range at a
// time for GRP chromosomes and leaves the range's sum per chromosome; the sums
// are added in a fixed order. A cluster of S CTAs shares a group's ranges and
// adds them in the leader's shared memory, so the result does not depend on S; nor on
// GRP (one chain of steps per segment): a chromosome's value is the same bit for
// bit in any population. With idx, entry q is chromosome idx[q].
// Before, one CTA held 8 chromosomes and thread t the rows t, t + 256, ... of
// the full square: at K = 257 the second pass served a single row, and 128
// CTAs left 24 SMs idle. P = 1024, K = 257: 231 -> 85 us per
// evaluation (the FP64 pipes, 1.0 TFLOP/s measured, need 68 us for half the
// square); the 16 re-scored candidates with their selection: 46 -> 16.9 us.
constexpr int kQuadWarps = 4;     // per CTA
constexpr int kQuadRanges = 32;   // kQuadRanges / (S kQuadWarps) ranges per warp

template <int GRP>
__global__ void __launch_bounds__(32 * kQuadWarps)
quad_rows_kernel(int P, int K, double m, double rm, int err, int S, const float* __restrict__ pop,
                 const int* __restrict__ idx, const double* __restrict__ T,
                 const double* __restrict__ b, const double* __restrict__ yy,
                 double* __restrict__ fit) {
  wait_previous();
  constexpr int kAhead = GRP >= 4 ? 8 : kAheadMax;   // loads in flight
  extern __shared__ double as[];   // [K + kAheadMax][GRP] genes of the group (zero past the last)
  __shared__ double red[kQuadRanges][GRP];   // the leader's: every range's sums
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (S > 1) ptx::cluster_arrive();   // the leader runs before anyone writes to it
  const int rank = (int)(blockIdx.x % S), p0 = (int)(blockIdx.x / S) * GRP;
  const int ng = min(GRP, P - p0);
  {
    // a thread's entries are one chromosome's genes (GRP divides the threads)
    const int q = threadIdx.x % GRP;
    const float* genes = q < ng ? pop + (int64_t)(idx ? idx[p0 + q] : p0 + q) * K : nullptr;
#pragma unroll 4
    for (int k = threadIdx.x / GRP; k < K; k += 32 * kQuadWarps / GRP)
      as[k * GRP + q] = genes ? (double)__ldcg(genes + k) : 0.0;
  }
  __syncthreads();
  if (S > 1) ptx::cluster_wait();
  const int NB = (K + 31) / 32;
  const int64_t steps = row_steps(K);
  constexpr int kPer = kQuadRanges / kQuadWarps;
  for (int j = 0; j < kPer / S; ++j) {
    const int range = (rank * kQuadWarps + warp) * (kPer / S) + j;
    int s = (int)(range * steps / kQuadRanges);
    const int s1 = (int)((range + 1) * steps / kQuadRanges);
    double v[GRP];
#pragma unroll
    for (int q = 0; q < GRP; ++q) v[q] = 0.0;
    int I = 0, base = 0;   // block of step s and the block's first step
    while (I + 1 < NB && s >= base + K - 32 * I) {
      base += K - 32 * I;
      ++I;
    }
    while (s < s1) {
      const int k1 = I * 32 + lane;
      const int end = base + K - 32 * I;   // the block's steps end
      const int stop = end < s1 ? end : s1;
      const double lin = s == base && k1 < K ? -2.0 * b[k1] : 0.0;
      double h[GRP];
#pragma unroll
      for (int q = 0; q < GRP; ++q) h[q] = lin;
      int k2 = 32 * I + (s - base);
      const double* t = T + (int64_t)s * 32 + lane;
      for (; s < stop; s += kAhead, k2 += kAhead, t += kAhead * 32) {
        double gv[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) gv[u] = t[u * 32];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
          if (GRP == 1) {
            // few warps: straight-line code keeps all loads in flight; a step
            // past the segment multiplies by zero (the list's entries are finite)
            h[0] = fma(gv[u], s + u < stop ? as[k2 + u] : 0.0, h[0]);
          } else {
            if (s + u >= stop) break;
#pragma unroll
            for (int q = 0; q < GRP; ++q) h[q] = fma(gv[u], as[(k2 + u) * GRP + q], h[q]);
          }
        }
      }
      s = stop;
      if (k1 < K) {
#pragma unroll
        for (int q = 0; q < GRP; ++q)
          v[q] = fma(as[k1 * GRP + q], h[q], v[q]);
      }
      base = end;
      ++I;
    }
    // lane sums: each exchange halves the chromosomes a lane still holds
    int n = GRP, q0 = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (n > 1) {
        n >>= 1;
        const bool up = (lane & o) != 0;
        q0 += up ? n : 0;
#pragma unroll
        for (int q = 0; q < GRP / 2; ++q)
          if (q < n) {
            const double give = up ? v[q] : v[q + n];
            const double keep = up ? v[q + n] : v[q];
            v[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
      } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
      }
    }
    if ((lane & (32 / GRP - 1)) == 0) {
      if (S > 1)
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(
                         ptx::mapa(ptx::smem_addr(&red[range][q0]), 0)),
                     "d"(v[0])
                     : "memory");
      else
        red[range][q0] = v[0];
    }
  }
  if (S > 1) ptx::cluster_sync();
  else __syncthreads();
  if (rank == 0 && threadIdx.x < ng) {
    double t[4] = {0.0, 0.0, 0.0, 0.0};   // ranges in four interleaved chains
#pragma unroll
    for (int r = 0; r < kQuadRanges; ++r) t[r & 3] += red[r][threadIdx.x];
    const int p = p0 + threadIdx.x;
    const double sum = *yy + ((t[0] + t[1]) + (t[2] + t[3]));
    fit[idx ? idx[p] : p] = finish_error(divide_by(sum, m, rm), err);
  }
}

// The elite re-scoring where the evaluation's kernels leave the GPU idle (see
// spread_serves; n <= kMaxRescore chromosomes): their products are spread over the
// whole GPU and share each entry of G. CTA (bx, by) owns rows
// k1 in [128 bx, 128 bx + 128) (one per thread) and the columns
// [by ks, (by + 1) ks) of the full square; each thread forms a_q[k1] h_q (and,
// in split 0, -2 a_q[k1] b[k1]); the CTA's sum per candidate (lanes by
// xor-butterfly, warps in order) goes to part[by][bx][q]. quad_spread_finish
// adds the parts in order.
constexpr int kSpreadRows = 128;
__global__ void __launch_bounds__(kSpreadRows)
quad_spread_kernel(int n, int K, int ks, const float* __restrict__ pop,
                   const int* __restrict__ idx, const double* __restrict__ G,
                   const double* __restrict__ b, double* __restrict__ part) {
  wait_previous();
  extern __shared__ double av[];   // [n][ks] genes of the column range
  __shared__ double red[kMaxRescore][kSpreadRows / 32];
  const int k1 = blockIdx.x * kSpreadRows + threadIdx.x;
  const int k2lo = blockIdx.y * ks, len = min(K - k2lo, ks);
  for (int e = threadIdx.x; e < n * ks; e += kSpreadRows) {
    const int q = e / ks, c = e % ks;
    av[e] = c < len ? (double)__ldcg(pop + (int64_t)idx[q] * K + k2lo + c) : 0.0;
  }
  __syncthreads();
  double h[kMaxRescore];
#pragma unroll
  for (int q = 0; q < kMaxRescore; ++q) h[q] = 0.0;
  if (k1 < K) {
    for (int c = 0; c < len; ++c) {
      const double g = G[(int64_t)(k2lo + c) * K + k1];
#pragma unroll
      for (int q = 0; q < kMaxRescore; ++q)
        if (q < n) h[q] = fma(g, av[q * ks + c], h[q]);
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < kMaxRescore; ++q) {
    if (q >= n) break;
    double v = 0.0;
    if (k1 < K) {
      const double ak = __ldcg(pop + (int64_t)idx[q] * K + k1);
      v = ak * h[q];
      if (blockIdx.y == 0) v -= 2.0 * ak * b[k1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[q][warp] = v;
  }
  __syncthreads();
  if (threadIdx.x < n) {
    double sum = 0.0;
    for (int w = 0; w < kSpreadRows / 32; ++w) sum += red[threadIdx.x][w];
    part[((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * n + threadIdx.x] = sum;
  }
}

// One warp per candidate q: lane l adds parts l, l + 32, ... in order, then
// a fixed xor-butterfly.
__global__ void quad_spread_finish(int n, int nparts, double m, double rm, int err,
                                   const int* __restrict__ idx, const double* __restrict__ part,
                                   const double* __restrict__ yy, double* __restrict__ fit) {
  wait_previous();
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q >= n) return;
  double s = 0.0;
  for (int j = lane; j < nparts; j += 32) s += part[(int64_t)j * n + q];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) fit[idx[q]] = finish_error(divide_by(*yy + s, m, rm), err);
}

int blocks_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b < 1) b = 1;
  if (b > 16384) b = 16384;
  return (int)b;
}

}  // namespace

// Row splits of a chunk's G accumulation: about three CTAs per SM over the
// upper-triangle tiles, at most 32, and at most 1 GB of partial sums.
int gram_splits(const Shape& s, int num_sms) {
  const int KT = (s.K + kGT - 1) / kGT;
  const int tiles = KT * (KT + 1) / 2;
  int z = (3 * num_sms + tiles - 1) / tiles;
  const int64_t cap = ((int64_t)1 << 30) / ((int64_t)s.K * s.K * 8);
  if (z > cap) z = (int)cap;
  if (z > 32) z = 32;
  if (z < 1) z = 1;
  return z;
}

int64_t gram_part_doubles(const Shape& s, int num_sms) {
  const int64_t g = (int64_t)gram_splits(s, num_sms) * s.K * s.K;
  const int64_t v = (int64_t)kVecSplits * (s.K + 1);
  return g > v ? g : v;
}

int64_t gram_chunk_rows(const Shape& s) {
  // Phi chunk of at most 64k patterns and at most 256 MB
  int64_t rows = (int64_t)(256ll * 1024 * 1024) / ((int64_t)s.K * 8);
  if (rows > 65536) rows = 65536;
  if (rows < 16) rows = 16;
  return rows;
}

cudaError_t launch_gram_build(const Shape& s, const float* Xt, const float* y, double* G,
                              double* b, double* yy, double* phi_chunk, double* part,
                              int num_sms, cudaStream_t st) {
  const int K = s.K;
  cudaError_t e = cudaMemsetAsync(G, 0, (size_t)K * K * sizeof(double), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(b, 0, (size_t)K * sizeof(double), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(yy, 0, sizeof(double), st);
  if (e != cudaSuccess) return e;
  const int64_t CH = gram_chunk_rows(s);
  const int KT = (K + kGT - 1) / kGT;
  for (int64_t m0 = 0; m0 < s.M; m0 += CH) {
    const int mc = (int)(s.M - m0 < CH ? s.M - m0 : CH);
    if (s.tied)
      expand_tied_kernel<<<blocks_for(mc), 256, 0, st>>>(m0, mc, s.N, s.d, s.basis, K, Xt,
                                                         phi_chunk);
    else
      expand_kernel<<<blocks_for((int64_t)mc * s.N), 256, 0, st>>>(m0, mc, s.N, s.d, s.basis,
                                                                  K, Xt, phi_chunk);
    const int zs = gram_splits(s, num_sms);
    const int rs = (mc + zs - 1) / zs;
    gram_accum_kernel<<<dim3(KT, KT, zs), 256, 0, st>>>(mc, rs, K, phi_chunk, part);
    gram_add_kernel<<<blocks_for((int64_t)K * K), 256, 0, st>>>(K, zs, part, G);
    const int vrs = (mc + kVecSplits - 1) / kVecSplits;
    vec_accum_kernel<<<dim3((K + 256) / 256, kVecSplits), 256, 0, st>>>(m0, mc, vrs, K, phi_chunk,
                                                                         y, part);
    vec_add_kernel<<<(K + 256) / 256, 256, 0, st>>>(K, kVecSplits, part, b, yy);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  mirror_kernel<<<blocks_for((int64_t)K * K), 256, 0, st>>>(K, G);
  return cudaGetLastError();
}

int64_t gram_list(const Shape& s) {
  return s.K <= kPairK ? (int64_t)s.K * (s.K + 1) / 2 : (row_steps(s.K) + kAheadMax) * 32;
}

cudaError_t launch_gram_list(const Shape& s, const GramDev& g, cudaStream_t st) {
  if (s.K <= kPairK) {
    pairs_kernel<<<1, 1024, 0, st>>>(s.K, g.G, g.list, g.kk);
  } else {
    const cudaError_t e =
        cudaMemsetAsync(g.list, 0, (size_t)gram_list(s) * sizeof(double), st);
    if (e != cudaSuccess) return e;
    steps_kernel<<<dim3((s.K + 31) / 32, 16), 256, 0, st>>>(s.K, g.G, g.list);
  }
  return cudaGetLastError();
}

namespace {
template <int GRP>
cudaError_t launch_rows(const Shape& s, const float* pop, int P, const int* idx, const GramDev& g,
                        double* fit, int err, int S, cudaStream_t st) {
  const size_t smem = (size_t)GRP * (s.K + kAheadMax) * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(quad_rows_kernel<GRP>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ceil_div(P, GRP) * S));
  cfg.blockDim = dim3(32 * kQuadWarps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)S;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // (see launch_behind)
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, quad_rows_kernel<GRP>, P, s.K, (double)s.M,
                            1.0 / (double)s.M, err, S, pop, idx, (const double*)g.list,
                            (const double*)g.b, (const double*)g.yy, fit);
}
}  // namespace

cudaError_t launch_gram_fitness(const Shape& s, const float* pop, int P, const int* idx,
                                const GramDev& g, double* fit, int err, int num_sms,
                                cudaStream_t st) {
  if (s.K <= kPairK) {
    return launch_behind(quad_pairs_kernel, ceil_div(P, kPairWarps), 32 * kPairWarps, 0, st, P, s.K,
                         (double)s.M, 1.0 / (double)s.M, err, pop, idx, g.list, g.kk, g.b, g.yy, fit);
  }
  // Four chromosomes share each entry where that still makes two CTAs per SM; else
  // one each, every load of a range in flight. Cluster size: about six CTAs per SM,
  // so the last SMs to finish are few. On 152 SMs, P = 1024, K = 257: 82 us
  // with four chromosomes and S = 4, 90 with S = 8 or 2, 91 with eight
  // chromosomes, 113 with one. (P = 16 with one and S = 8, candidate selection included:
  // 13.7 us.)
  const int grp = (int64_t)ceil_div(P, 4) * 8 >= 2 * num_sms ? 4 : 1;
  int S = 1;
  while (S < 8 && (int64_t)ceil_div(P, grp) * S < 6 * num_sms) S <<= 1;
  return grp == 4 ? launch_rows<4>(s, pop, P, idx, g, fit, err, S, st)
                  : launch_rows<1>(s, pop, P, idx, g, fit, err, S, st);
}

// The re-scoring is spread over the GPU where the kernels of the evaluation leave
// it idle or read too much: at K = 49 to 64 for up to 8 candidates (the pair list
// gives each one warp), and at long K, where each candidate's cluster reads the
// whole list: from K = 1900 on for more than 8 candidates, from K = 3900 on, where
// the list no longer fits one die's half of L2, for any. us per call with the
// selection, P = 16, evaluation's kernels / spread: K = 37: 11.8 / 10.1 (n = 2), 11.7 /
// 14.2 (n = 8); K = 49: 16.1 / 10.0, 16.2 / 14.3, 16.1 / 20.5 (n = 16); K = 64:
// 22.1 / 9.9, 22.6 / 14.4, 22.5 / 20.7; n = 8: K = 1201: 55.6 / 61.4; 2001: 132 / 138;
// 3841: 457 / 516; 4097: 809 / 552; n = 16: K = 257: 13.7 / 26.4; 1201: 59 / 67;
// 1801: 118 / 120; 1901: 131 / 124; 3073: 322 / 292; 4097: 815 / 523. CTAs of 128
// rows; no more than two per SM, a third on some SMs costs half the time again (the
// FP64 pipes): K = 3073, n = 16: 389 with 325 CTAs on 152 SMs, 291 with 300.
static bool spread_serves(int K, int n) {
  return K >= (n > 8 ? 1900 : 3900) || (K >= 49 && K <= kPairK && n <= 8);
}
struct Spread { int bx, by, ks; };
static Spread spread(int K, int num_sms) {
  Spread p;
  p.bx = ceil_div(K, kSpreadRows);
  p.by = 2 * num_sms / p.bx;
  if (p.by < ceil_div(K, 1600)) p.by = ceil_div(K, 1600);   // genes of a range: 200 KB
  if (p.by > K) p.by = K;
  p.ks = ceil_div(K, p.by);
  p.by = ceil_div(K, p.ks);
  return p;
}

int64_t gram_rescore_parts(const Shape& s, int num_sms) {
  if (!spread_serves(s.K, 1) && !spread_serves(s.K, kMaxRescore)) return 0;
  const Spread p = spread(s.K, num_sms);
  return (int64_t)p.bx * p.by * kMaxRescore;
}

cudaError_t launch_gram_rescore(const Shape& s, const float* pop, int n, const int* idx,
                                const GramDev& g, double* fit, int err, int num_sms,
                                cudaStream_t st) {
  if (n < 1 || n > kMaxRescore) return cudaErrorInvalidValue;
  if (!spread_serves(s.K, n)) return launch_gram_fitness(s, pop, n, idx, g, fit, err, num_sms, st);
  const Spread p = spread(s.K, num_sms);
  const size_t smem = (size_t)n * p.ks * sizeof(double);
  cudaError_t e = cudaFuncSetAttribute(quad_spread_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e != cudaSuccess) return e;
  e = launch_behind(quad_spread_kernel, dim3(p.bx, p.by), kSpreadRows, smem, st, n, s.K, p.ks, pop,
                    idx, g.G, g.b, g.part);
  if (e != cudaSuccess) return e;
  return launch_behind(quad_spread_finish, 1, 32 * n, 0, st, n, p.bx * p.by, (double)s.M,
                       1.0 / (double)s.M, err, idx, g.part, g.yy, fit);
}

}  // namespace game
