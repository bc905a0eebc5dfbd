// tc_common.cuh -- device helpers shared by the tensor-core fitness kernels
// (single problem and batched): bounded mbarrier waits, the fused
// squared- or absolute-error epilogue step, and operand rounding to BF16 /
// E4M3.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <stdint.h>

#include "game_internal.cuh"
#include "tc_ptx.cuh"

namespace game {
namespace tc {

// Limit of one wait, in cycles of the SM: 1.9 s at its highest clock (2070 MHz), 2.8 s
// at the 1.45 GHz of long loads under the power cap. (The global timer, which would
// give seconds, costs microseconds to read.)
constexpr long long kTimeoutCycles = 4000000000ll;
constexpr uint32_t kSuspendNs = 20000;           // per try_wait suspension (woken early on completion)

// Bounded wait for the phase of the given parity. Waiting threads are
// suspended by the hardware (suspend-time hint) instead of spinning, so they
// take no issue slots from the MMA issuer and the producers on their SM
// sub-partition; each wake-up re-checks the abort flag and the time limit.
static __device__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status) {
  if (ptx::mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
    if (ptx::mbar_try_wait_sleep(bar, parity, kSuspendNs)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > kTimeoutCycles) {
      *abort_flag = 1;
      atomicExch(status, (int)kDevTimeout);
      return false;
    }
  }
}

// Waits for this CTA's own asynchronous work (copies, MMAs) regardless of the
// abort flag, still bounded.
static __device__ void wait_bar_drain(uint32_t bar, uint32_t parity, int* status) {
  const long long t0 = clock64();
  while (!ptx::mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > kTimeoutCycles) {
      atomicExch(status, (int)kDevTimeout);
      return;
    }
  }
}

// ---- epilogue of the population-sized kernels ----
// What bounds it: an accumulator of 256 patterns is due every 16 K' tensor
// cycles (2048 at K' = 256), in which each of the eight warps reduces 32 rows x
// 128 columns; its latencies (tensor memory, the targets from a shared memory
// that the MMAs read at the same time, the FP64 sums, the bias) are of the same
// length, so each is started one step ahead of its use. BF16, M = 10^6, N = 32,
// degree 8, P = 1024: 355 us per evaluation without, 340 with.

// targets of 16 columns; YS: they are in shared memory (else global memory,
// read through the read-only path)
template <bool YS>
__device__ __forceinline__ void epi_targets(const float* yc, float4 (&y)[4]) {
#pragma unroll
  for (int e4 = 0; e4 < 4; ++e4)
    y[e4] = YS ? reinterpret_cast<const float4*>(yc)[e4]
               : __ldg(reinterpret_cast<const float4*>(yc) + e4);
}

// sse += ((y - bias) - u * acc)^2 over 16 columns, two columns per packed op
// (ABS: += |(y - bias) - u * acc|, the absolute error).
// SCALED = false: u = 1 and the residual is one packed subtraction; true
// (FP8): -u * acc + (y - bias) as one packed FMA (one rounding, as the
// subtraction is for u = 1).
template <bool SCALED, bool ABS>
__device__ __forceinline__ void epi_cols16(const uint32_t (&v)[16], const float4 (&y)[4],
                                           uint64_t bias2, uint64_t negu2, uint64_t& s2) {
#pragma unroll
  for (int e4 = 0; e4 < 4; ++e4) {
    const uint64_t ya = ptx::f2_sub(ptx::f2_pack(y[e4].x, y[e4].y), bias2);
    const uint64_t yb = ptx::f2_sub(ptx::f2_pack(y[e4].z, y[e4].w), bias2);
    const uint64_t da = ptx::f2_pack(__uint_as_float(v[4 * e4]), __uint_as_float(v[4 * e4 + 1]));
    const uint64_t db = ptx::f2_pack(__uint_as_float(v[4 * e4 + 2]), __uint_as_float(v[4 * e4 + 3]));
    const uint64_t ra = SCALED ? ptx::f2_fma(negu2, da, ya) : ptx::f2_sub(ya, da);
    const uint64_t rb = SCALED ? ptx::f2_fma(negu2, db, yb) : ptx::f2_sub(yb, db);
    if (ABS) {
      s2 = ptx::f2_add(s2, ptx::f2_abs(ra));
      s2 = ptx::f2_add(s2, ptx::f2_abs(rb));
    } else {
      s2 = ptx::f2_fma(ra, ra, s2);
      s2 = ptx::f2_fma(rb, rb, s2);
    }
  }
}

// One thread's sums of the last accumulator: turned into FP64 and added to the
// running sum in two pieces of the next accumulator's reduction (begin ahead of
// its wait, end behind its first load).
struct LastSum {
  float2 sum = {0.f, 0.f};
  float tail = 0.f;
  double* row = nullptr;   // the running sum's place
  bool first = false;      // nothing there yet
  double sse = 0.0, before = 0.0;
  __device__ __forceinline__ void begin() {
    if (!row) return;
    before = first ? 0.0 : *row;
    sse = (double)sum.x + (double)sum.y;
    if (tail != 0.f) sse += (double)tail;   // (FP64 operations are scarce)
  }
  __device__ __forceinline__ void end() {
    if (row) *row = first ? sse : before + sse;
  }
};

// The sums of `valid` columns (a multiple of 32 but in the last tile)
// of this thread's row at tensor-memory address tbase. ya: the first 16
// columns' targets (epi_targets), where valid >= 32. 16 columns at a time, the
// next load in flight (by 32 the registers spill).
template <bool SCALED, bool ABS, bool YS>
__device__ __forceinline__ void epi_reduce(uint32_t tbase, const float* yt, int valid,
                                           float4 (&ya)[4], float bias, float negu, LastSum& last,
                                           float2& sum, float& tail) {
  const uint64_t bias2 = ptx::f2_pack(bias, bias), negu2 = ptx::f2_pack(negu, negu);
  const int nfull = valid / 32;
  uint64_t s2 = 0;   // two FP32 partial sums (even / odd columns)
  tail = 0.f;
  if (nfull > 0) {
    float4 yb[4];
    uint32_t va[16], vb[16];
    ptx::tmem_ld16_issue(tbase, va);
    ptx::tmem_ld16_wait(va);
    last.end();
    for (int k = 0; k < 2 * nfull; k += 2) {
      ptx::tmem_ld16_issue(tbase + (uint32_t)(k + 1) * 16, vb);
      epi_targets<YS>(yt + k * 16 + 16, yb);
      epi_cols16<SCALED, ABS>(va, ya, bias2, negu2, s2);
      ptx::tmem_ld16_wait(vb);
      const bool more = k + 2 < 2 * nfull;
      if (more) {
        ptx::tmem_ld16_issue(tbase + (uint32_t)(k + 2) * 16, va);
        epi_targets<YS>(yt + k * 16 + 32, ya);
      }
      epi_cols16<SCALED, ABS>(vb, yb, bias2, negu2, s2);
      if (more) ptx::tmem_ld16_wait(va);
    }
  } else {
    last.end();
  }
  if (nfull * 32 < valid) {   // ragged last columns of the last tile
    uint32_t v[32];
    ptx::tmem_ld32(tbase + (uint32_t)nfull * 32, v);
    const int lim = valid - nfull * 32;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      if (e < lim) {
        const float r = SCALED ? fmaf(negu, __uint_as_float(v[e]), yt[nfull * 32 + e] - bias)
                               : (yt[nfull * 32 + e] - bias) - __uint_as_float(v[e]);
        tail = ABS ? tail + fabsf(r) : fmaf(r, r, tail);
      }
    }
  }
  sum = ptx::f2_unpack(s2);
}

// Rounds 2 x 8 values to BF16 pairs (hi), and for bf16x3 also the residuals
// v - hi (lo).
__device__ __forceinline__ uint32_t bf16x2_bits(float lo_col, float hi_col) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo_col, hi_col);
  return *reinterpret_cast<const uint32_t*>(&b);
}
__device__ __forceinline__ void split_bf16x2(float v0, float v1, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
  const float2 hf = __bfloat1622float2(h);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = bf16x2_bits(v0 - hf.x, v1 - hf.y);
}
__device__ __forceinline__ uint32_t e4m3x4_bits(float v0, float v1, float v2, float v3) {
  const uint32_t lo = __nv_cvt_float2_to_fp8x2(make_float2(v0, v1), __NV_SATFINITE, __NV_E4M3);
  const uint32_t hi = __nv_cvt_float2_to_fp8x2(make_float2(v2, v3), __NV_SATFINITE, __NV_E4M3);
  return lo | (hi << 16);
}

}  // namespace tc
}  // namespace game
