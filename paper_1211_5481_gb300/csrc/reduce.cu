// reduce.cu -- cross-tile FP64 error sum: fit[p] = (sum_r part[r][p]) / M
// (the MSE from squared residuals, the MAE from absolute ones), or its square
// root for the RMSE.
//
// What bounds it: the FP64 adders of the SMs in use (an SM does two adds a
// cycle: the 304 rows of 1024 chromosomes on 32 SMs take 2.4 us) and latency.
// So a CTA takes only 8 chromosomes: 8 neighbouring lanes read a row's 64
// bytes, 32 row groups r, r + 32, ... are added in order with their loads in
// flight together, and the groups' sums in four interleaved chains. The order
// depends only on the number of rows, so the result is bit-identical run to
// run (no atomics). One warp per chromosome, lanes striding over the rows,
// touched 32 sectors per load: 5.7 us at P = 1024, 304 rows; this 5.3.
#include "fp64.cuh"
#include "game_internal.cuh"

namespace game {

namespace {

constexpr int kChroms = 8, kGroups = 32;   // per CTA; a thread each

__global__ void __launch_bounds__(kChroms * kGroups)
reduce_rows_kernel(const double* __restrict__ part, int rows, int P, int Ppad, int err, double m,
                   double rm, double* __restrict__ fit) {
  __shared__ double sum[kGroups][kChroms];
  wait_previous();
  const int c = threadIdx.x % kChroms, grp = threadIdx.x / kChroms;
  const int p = blockIdx.x * kChroms + c;   // Ppad is a multiple of 128: in bounds past P
  double s = 0.0;
  for (int r0 = grp; r0 < rows; r0 += 10 * kGroups) {
    double v[10];
#pragma unroll
    for (int u = 0; u < 10; ++u) {
      const int r = r0 + u * kGroups;
      v[u] = r < rows ? part[(int64_t)r * Ppad + p] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 10; ++u)
      if (r0 + u * kGroups < rows) s += v[u];
  }
  sum[grp][c] = s;
  __syncthreads();
  if (grp != 0 || p >= P) return;
  double t[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) t[k] = sum[k][c];
  for (int k = 4; k < kGroups && k < rows; k += 4) {
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] += sum[k + j][c];
  }
  const double mean = divide_by((t[0] + t[1]) + (t[2] + t[3]), m, rm);
  fit[p] = err == GAME_ERR_RMSE ? sqrt(mean) : mean;
}

}  // namespace

cudaError_t launch_reduce(const double* part, int rows, int P, int Ppad, int64_t M, int err,
                          double* fit, cudaStream_t st) {
  return launch_behind(reduce_rows_kernel, ceil_div(P, kChroms), kChroms * kGroups, 0, st, part,
                       rows, P, Ppad, err, (double)M, 1.0 / (double)M, fit);
}

}  // namespace game
