// gram.cuh -- device pieces of the Gram form shared by its kernels (gram.cu)
// and by the whole-generation kernel of small runs (gram_train.cu): one
// chromosome's value is the same bit for bit wherever it is computed.
#pragma once
#include <math_constants.h>
#include <stdint.h>

#include "fp64.cuh"
#include "game_internal.cuh"
#include "tc_ptx.cuh"

namespace game {

constexpr int kPairK = 64;   // genes up to which the pair list serves

// The fitness from the Gram-form MSE, clamped at 0 (cancellation can leave
// an exact fit a few ulps below zero): itself, or its square root for
// GAME_ERR_RMSE.
__device__ __forceinline__ double finish_error(double mse, int err) {
  const double m = fmax(mse, 0.0);
  return err == GAME_ERR_RMSE ? sqrt(m) : m;
}

// a^T G a - 2 a.b of one chromosome by one warp, genes a [K] FP64 in shared
// memory, Gp / kk the weighted pair list: lane l takes entries l, l + 32, ...
// in two interleaved sums, then genes l, l + 32, ..., then a fixed
// xor-butterfly; every lane gets it.
// (Lane = row of the full square costs K steps of K / 32 partly filled warps;
// the list K^2 / 64 full ones, two FP64 operations each. FP64 latency decides
// at these sizes: eight entries' loads and products are in flight together.)
__device__ __forceinline__ double quad_pairs(int K, const double* a, const double* Gp,
                                             const uint16_t* kk, const double* b, int lane) {
  double v0 = 0.0, v1 = 0.0, w = 0.0;
  const int E = K * (K + 1) / 2;
  for (int k = lane; k < K; k += 32) w = fma(-2.0 * a[k], b[k], w);
  for (int e0 = lane; e0 < E; e0 += 256) {
    double t[8], g[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + 32 * u;
      const int k = e < E ? kk[e] : 0;
      g[u] = e < E ? Gp[e] : 0.0;
      t[u] = e < E ? a[k & 255] * a[k >> 8] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      if (e0 - lane + 32 * u >= E) break;
      v0 = fma(g[u], t[u], v0);
      v1 = fma(g[u + 1], t[u + 1], v1);
    }
  }
  double v = (v0 + v1) + w;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace game
