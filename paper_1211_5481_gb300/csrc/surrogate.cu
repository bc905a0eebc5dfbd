// surrogate.cu -- a small MLP that predicts a chromosome's fitness, trained
// online on the (chromosome, exact fitness) pairs the GA produces, and used to
// screen oversampled offspring so that only the most promising get the exact
// fitness of paper Section 3 (Eq. 2, Eq. 3).
//
// Network: x in R^K (the genes) -> 256 -> 256 -> 1. Layers 1 and 2 take BF16
// operands (inputs, weights and the layer-1 activations rounded to BF16) with
// FP32 accumulation; the output layer is FP32. Activation: GELU in its tanh
// form, g(z) = z/2 (1 + tanh(c (z + 0.044715 z^3))), c = sqrt(2/pi). Target:
// the log-fitness l = log(max(fit, 1e-30)) standardised over the training
// batch, t = (l - mean l) / sd l (FP64 statistics; sd 0 counts as 1): the
// MSE spans orders of magnitude and only the ranking of the prediction is
// used. Loss: mean of (out - t)^2 over the batch. Optimiser: Adam (lr 1e-3, beta1 0.9, beta2 0.999, eps 1e-8) on FP32
// master weights. Initial weights uniform in +-1/sqrt(fan_in) from
// Philox4x32-10 (key = seed, counter = (layer, index, 0, tag 9)), biases 0.
//
// Parameter vector (FP32, this order): W1 [256][K], b1 [256], W2 [256][256],
// b2 [256], w3 [256], b3 [1].
//
// Kernels. The products whose operands lie along k in memory -- X W1^T, H1 W2^T
// and dZ2 W2 -- take BF16 copies of them (gemm_nt_kernel: all K-blocks copied
// asynchronously at once, no conversion on the way; Adam refreshes the weights'
// copies, the batch's is made once per batch). The weight gradients (reduction
// over the batch) take FP32 operands, transposed on the way and split into BF16
// hi + lo (grad_gemm_kernel, split-K, both layers in one launch). Between them:
// one kernel for the output layer, its gradient and dZ2, one for the four bias
// and output-weight sums, one for the split sums and Adam. A training step is
// seven launches. With conversion inside one generic GEMM, the statistics of
// the batch in every step and a kernel per elementwise step it was 19: 178 us a
// step at P = 2048, K = 289, now 60.
// Screening: a radix selection of the predictions in one CTA that also numbers
// the kept slots, and a gather in slot order (19 us; sorting and compacting took 223). The exact
// fitness checks the surrogate: after each screened generation the Pearson
// correlation r of the kept children's predictions with their exact
// log-fitness is measured, and the next screening trusts the surrogate only
// if r > 0.25; otherwise it keeps the first P - E children, i.e. exactly the
// children of the unscreened generation.
#include <cuda_bf16.h>

#include "game_internal.cuh"
#include "philox.cuh"
#include "tc_ptx.cuh"

namespace game {

namespace {

constexpr int kH = kSurrogateHidden;
constexpr float kGeluC = 0.7978845608028654f;   // sqrt(2 / pi)
constexpr float kGeluA = 0.044715f;

__device__ __forceinline__ float gelu(float z) {
  const float u = kGeluC * (z + kGeluA * z * z * z);
  return 0.5f * z * (1.f + tanhf(u));
}

__device__ __forceinline__ float gelu_grad(float z) {
  const float u = kGeluC * (z + kGeluA * z * z * z);
  const float t = tanhf(u);
  return 0.5f * (1.f + t) + 0.5f * z * (1.f - t * t) * kGeluC * (1.f + 3.f * kGeluA * z * z);
}

// Waits are bounded (1 s): an expired wait abandons the tile and raises
// *status.
constexpr int kGTK = 64;                  // K per block (128 bytes of BF16 per row)
constexpr uint32_t kGemmWaitNs = 1000000000ull;

__device__ __forceinline__ bool g_wait(uint32_t bar, uint32_t parity, int* status) {
  if (ptx::mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = ptx::global_timer_ns();
  while (!ptx::mbar_try_wait(bar, parity))
    if (ptx::global_timer_ns() - t0 > kGemmWaitNs) {
      atomicExch(status, (int)kDevTimeout);
      return false;
    }
  return true;
}

__device__ __forceinline__ uint32_t bf16pair(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&b);
}

// 8 consecutive k of one row into the swizzled image (hi, and lo when split)
__device__ __forceinline__ void g_store8(uint8_t* img, uint8_t* img_lo, int r, int qd,
                                         const float (&v)[8], bool split) {
  const int off = r * 128 + ((qd ^ (r & 7)) << 4);
  uint32_t h[4], l[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    h[e] = bf16pair(v[2 * e], v[2 * e + 1]);
    if (split) {
      const __nv_bfloat162 hb = *reinterpret_cast<const __nv_bfloat162*>(&h[e]);
      const float2 hf = __bfloat1622float2(hb);
      l[e] = bf16pair(v[2 * e] - hf.x, v[2 * e + 1] - hf.y);
    }
  }
  *reinterpret_cast<uint4*>(img + off) = make_uint4(h[0], h[1], h[2], h[3]);
  if (split) *reinterpret_cast<uint4*>(img_lo + off) = make_uint4(l[0], l[1], l[2], l[3]);
}

// Rows [0, R) x k in [k0, k0 + 64) of an operand X(r, k) = X[(r0 + r) + k ks] (zero
// where r0 + r >= rlim or k >= kend) into the swizzled image, by the CTA's
// kGThreads threads: consecutive threads take consecutive rows (a warp's loads
// span 32 rows), the row's eight 16-byte units split among kGThreads / R threads.
// Every thread issues all of its loads before it converts and stores anything, so
// each waits one memory latency per K-block.
constexpr int kGThreads = 256;
template <int R>
__device__ __forceinline__ void g_load(uint8_t* img, uint8_t* img_lo, const float* __restrict__ X,
                                       int64_t ks, int r0, int rlim, int k0, int kend,
                                       bool split) {
  constexpr int TPR = kGThreads / R;              // threads per row
  constexpr int UPT = 8 / TPR;                    // units per thread
  const int tid = threadIdx.x, r = tid % R, ug = tid / R, row = r0 + r;
  float v[UPT][8];
#pragma unroll
  for (int u = 0; u < UPT; ++u)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = k0 + (ug * UPT + u) * 8 + e;
      v[u][e] = (row < rlim && k < kend) ? X[(int64_t)row + (int64_t)k * ks] : 0.f;
    }
#pragma unroll
  for (int u = 0; u < UPT; ++u) g_store8(img, img_lo, r, ug * UPT + u, v[u], split);
}

constexpr int kGTN = 64;   // columns of C per CTA

// One weight gradient: C[m][n] = sum_b A[b][m] B[b][n] (A = dZ [batch][256] FP32
// entering as BF16 hi + lo, B = the layer's input [batch][N] rounded to BF16).
struct GradProblem {
  const float *A, *B;
  float* parts;   // [splits][256][N] partial products
  int N, tiles;   // column tiles of kGTN
};

// Both layers' weight gradients in one launch: blockIdx.x < p0.tiles is the
// first problem's column tile, the rest the second's; blockIdx.y the 128-row
// tile of the 256 outputs; blockIdx.z takes batch rows [z kz, (z + 1) kz) and
// writes its partial product to parts + z 256 N (added in order by adam_kernel).
// Products: hi hi + lo hi.
__global__ void __launch_bounds__(kGThreads, 1)
grad_gemm_kernel(int batch, GradProblem p0, GradProblem p1, int kz, int* status) {
  wait_previous();
  constexpr uint32_t kAImg = 128 * 128, kBImg = kGTN * 128;
  constexpr uint32_t kStage = 2 * kAImg + kBImg;   // hi and lo images of A
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + 2 * kStage);   // [2] stage free, [1] done
  uint32_t* holder = reinterpret_cast<uint32_t*>(bars + 3);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool first = (int)blockIdx.x < p0.tiles;
  const GradProblem p = first ? p0 : p1;
  const int n0 = (first ? (int)blockIdx.x : (int)blockIdx.x - p0.tiles) * kGTN;
  const int m0 = blockIdx.y * 128;
  const int kbeg = blockIdx.z * kz;
  const int kend = min(batch, kbeg + kz);
  const int nkb = kend > kbeg ? (kend - kbeg + kGTK - 1) / kGTK : 0;
  if (tid == 0) {
    for (int b = 0; b < 3; ++b) ptx::mbar_init(ptx::smem_addr(&bars[b]), 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_addr(holder), kGTN);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *holder;
  const uint32_t idesc = ptx::idesc_bf16_f32(128, kGTN);
  bool ok = true;
  for (int kb = 0; kb < nkb && ok; ++kb) {
    const int st = kb & 1;
    uint8_t* a_img = base + st * kStage;
    uint8_t* a_lo = a_img + kAImg;
    uint8_t* b_img = a_img + 2 * kAImg;
    // the MMAs that read this stage two blocks ago are done
    if (kb >= 2) ok = g_wait(ptx::smem_addr(&bars[st]), ((kb - 2) >> 1) & 1, status);
    if (!ok) break;
    const int k0 = kbeg + kb * kGTK;
    g_load<128>(a_img, a_lo, p.A, kH, m0, kH, k0, kend, true);
    g_load<kGTN>(b_img, nullptr, p.B, p.N, n0, p.N, k0, kend, false);
    ptx::fence_proxy_async_smem();
    __syncthreads();
    if (tid == 0) {
      ptx::tc_fence_after();
      const uint64_t ad = ptx::desc_kmajor_sw128(ptx::smem_addr(a_img));
      const uint64_t adl = ptx::desc_kmajor_sw128(ptx::smem_addr(a_lo));
      const uint64_t bd = ptx::desc_kmajor_sw128(ptx::smem_addr(b_img));
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        const uint32_t o = 2u * ks;
        ptx::mma_bf16(tmem, ad + o, bd + o, idesc, (kb | ks) != 0);
        ptx::mma_bf16(tmem, adl + o, bd + o, idesc, 1u);
      }
      ptx::mma_commit(ptx::smem_addr(&bars[st]));
    }
  }
  // all MMAs done
  if (tid == 0) ptx::mma_commit(ptx::smem_addr(&bars[2]));
  const bool done = g_wait(ptx::smem_addr(&bars[2]), 0, status);
  ptx::tc_fence_after();
  // (the epilogue's scratch is the operand ring: every MMA of the CTA is done)
  if (__syncthreads_and(done && ok)) {
    // each warp's 32 accumulator rows go through a 32 x 33 scratch tile so that
    // the stores run along rows of C; warp w reads tensor-memory lanes
    // 32 (w % 4) .. (its quadrant), columns of half w / 4
    float* stage = reinterpret_cast<float*>(base) + warp * (32 * 33);
    float* Cz = p.parts + (int64_t)blockIdx.z * kH * p.N;
    const int quad = warp & 3, c0 = (warp >> 2) * (kGTN / 2);
    uint32_t v[32];
    ptx::tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
    for (int e = 0; e < 32; ++e) stage[lane * 33 + e] = nkb > 0 ? __uint_as_float(v[e]) : 0.f;
    __syncwarp();
    const int n = n0 + c0 + lane;
#pragma unroll 4
    for (int r = 0; r < 32; ++r)
      if (n < p.N) Cz[(int64_t)(m0 + quad * 32 + r) * p.N + n] = stage[r * 33 + lane];
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, kGTN);
  }
}

// C[m][n] = sum_k A[m][k] B[n][k] for M rows and N = 256 columns, A [M][lda]
// and B [256][lda] BF16, lda = nkb 64 (zero-padded), rows 16-byte aligned; with
// NA = 2 A is a hi + lo pair (products hi B, lo B). What bounds it: latency
// (2048 x 256 x 320 is a microsecond of tensor work over 64 CTAs), so a CTA
// starts the copies of all its K-blocks (up to kNtStages; a ring beyond) before
// it waits for the first. Epilogue:
//   kLayer  Z = C + bias; H = g(Z); keep != 0: Z and H to memory (FP32, H rounded
//           to BF16 where Hb is given); Hb the BF16 copy of H
//   kDelta  out = C g'(Zin)
enum NtMode : int { kLayer = 0, kDelta = 1 };
struct NtArgs {
  int M, nkb, mode, keep;
  const __nv_bfloat16 *A, *A2, *B;
  const float* bias;     // kLayer
  const float* Zin;      // kDelta
  float *Z, *H;          // kLayer (kDelta: H = out)
  __nv_bfloat16* Hb;
  int* status;
};
constexpr int kNtStages = 5;

template <int NA>
__host__ __device__ constexpr int nt_stages() { return NA == 1 ? kNtStages : 4; }
template <int NA>
__host__ __device__ constexpr int nt_smem() {
  return nt_stages<NA>() * (NA * 128 * 128 + kGTN * 128) + 1024 + 128;
}

template <int NA>
__global__ void __launch_bounds__(kGThreads, 1) gemm_nt_kernel(const NtArgs a) {
  wait_previous();
  constexpr int NS = nt_stages<NA>();
  constexpr uint32_t kAImg = 128 * 128;
  constexpr uint32_t kStage = NA * kAImg + kGTN * 128;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + NS * kStage);   // [NS] free, [1] done
  uint32_t* holder = reinterpret_cast<uint32_t*>(bars + NS + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * 128, n0 = blockIdx.x * kGTN;
  const int64_t lda = (int64_t)a.nkb * kGTK;
  if (tid == 0) {
    for (int b = 0; b <= NS; ++b) ptx::mbar_init(ptx::smem_addr(&bars[b]), 1);
    ptx::fence_mbar_init();
  }
  if (warp == 0) {
    ptx::tmem_alloc(ptx::smem_addr(holder), kGTN);
    ptx::tmem_relinquish();
  }
  // K-block kb into its stage: 16-byte units in the swizzled K-major layout,
  // rows past M zero; one commit group (empty past the last K-block)
  auto load = [&](int kb) {
    if (kb < a.nkb) {
      const uint32_t img = ptx::smem_addr(base + (kb % NS) * kStage);
      const int unit = tid & 7;
#pragma unroll
      for (int im = 0; im < NA; ++im) {
        const __nv_bfloat16* src = im ? a.A2 : a.A;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const int r = (tid >> 3) + 32 * p;
          const int row = m0 + r < a.M ? m0 + r : 0;
          ptx::cp_async16_zfill(img + im * kAImg + r * 128 + ((unit ^ (r & 7)) << 4),
                                src + row * lda + kb * kGTK + unit * 8, m0 + r < a.M);
        }
      }
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const int r = (tid >> 3) + 32 * p;
        ptx::cp_async16_zfill(img + NA * kAImg + r * 128 + ((unit ^ (r & 7)) << 4),
                              a.B + (n0 + r) * lda + kb * kGTK + unit * 8, true);
      }
    }
    ptx::cp_async_commit();
  };
#pragma unroll
  for (int kb = 0; kb < NS; ++kb) load(kb);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *holder;
  const uint32_t idesc = ptx::idesc_bf16_f32(128, kGTN);
  bool ok = true;
  for (int kb = 0; kb < a.nkb; ++kb) {
    ptx::cp_async_wait<NS - 1>();
    ptx::fence_proxy_async_smem();
    __syncthreads();
    const int st = kb % NS;
    if (tid == 0) {
      ptx::tc_fence_after();
      const uint64_t ad = ptx::desc_kmajor_sw128(ptx::smem_addr(base + st * kStage));
      const uint64_t bd = ptx::desc_kmajor_sw128(ptx::smem_addr(base + st * kStage + NA * kAImg));
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        const uint32_t o = 2u * ks;
        ptx::mma_bf16(tmem, ad + o, bd + o, idesc, (kb | ks) != 0);
        if (NA == 2) ptx::mma_bf16(tmem, ad + (kAImg >> 4) + o, bd + o, idesc, 1u);
      }
      ptx::mma_commit(ptx::smem_addr(&bars[st]));
    }
    if (kb + NS < a.nkb) ok = ok && g_wait(ptx::smem_addr(&bars[st]), (kb / NS) & 1, a.status);
    load(ok ? kb + NS : a.nkb);   // refilled once its MMAs are done
  }
  if (tid == 0) ptx::mma_commit(ptx::smem_addr(&bars[NS]));
  const bool done = g_wait(ptx::smem_addr(&bars[NS]), 0, a.status);
  ptx::cp_async_wait<0>();
  ptx::tc_fence_after();
  if (__syncthreads_and(done && ok)) {
    float* stage = reinterpret_cast<float*>(base) + warp * (32 * 33);
    const int quad = warp & 3, c0 = (warp >> 2) * (kGTN / 2);
    uint32_t v[32];
    ptx::tmem_ld32(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
    for (int e = 0; e < 32; ++e) stage[lane * 33 + e] = __uint_as_float(v[e]);
    __syncwarp();
    const int n = n0 + c0 + lane;
    const float bias = a.mode == kLayer ? a.bias[n] : 0.f;
#pragma unroll 4
    for (int r = 0; r < 32; ++r) {
      const int m = m0 + quad * 32 + r;
      if (m >= a.M) break;
      const int64_t at = (int64_t)m * kH + n;
      float x = stage[r * 33 + lane];
      if (a.mode == kLayer) {
        x += bias;
        const float g = gelu(x);
        if (a.keep) a.Z[at] = x;
        if (a.Hb) {
          const __nv_bfloat16 gb = __float2bfloat16_rn(g);
          a.Hb[at] = gb;
          if (a.keep) a.H[at] = __bfloat162float(gb);
        } else {
          a.H[at] = g;
        }
      } else {
        a.H[at] = x * gelu_grad(a.Zin[at]);
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, kGTN);
  }
}

// Xb [B][Kq] = X [B][K] rounded to BF16, zero past K (16-byte units).
__global__ void to_bf16_kernel(int64_t B, int K, int Kq, const float* __restrict__ X,
                               __nv_bfloat16* __restrict__ Xb) {
  wait_previous();
  const int per = Kq / 8;
  const int64_t n = B * per;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = e / per;
    const int k0 = (int)(e - b * per) * 8;
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = k0 + u < K ? __ldcg(X + b * K + k0 + u) : 0.f;
    reinterpret_cast<uint4*>(Xb)[e] = make_uint4(bf16pair(v[0], v[1]), bf16pair(v[2], v[3]),
                                                 bf16pair(v[4], v[5]), bf16pair(v[6], v[7]));
  }
}

// Output layer: out[b] = sum_j H2[b][j] w3[j] + b3, one warp per row, fixed lane
// order.
__device__ __forceinline__ float output_row(const float* __restrict__ H2,
                                            const float* __restrict__ w3, float b3, int lane) {
  float s = 0.f;
#pragma unroll
  for (int j = 0; j < kH; j += 32) s = fmaf(H2[j + lane], w3[j + lane], s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s + b3;
}

__global__ void output_kernel(int B, const float* __restrict__ H2, const float* __restrict__ w3,
                              const float* __restrict__ b3, float* __restrict__ out) {
  wait_previous();
  const int w = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= B) return;
  const float s = output_row(H2 + (int64_t)w * kH, w3, b3[0], lane);
  if (lane == 0) out[w] = s;
}

// A training row: the output, d_out[b] = 2 (out[b] - t[b]) / B, the loss term
// (out - t)^2 / B, and dZ2[b][j] = d_out[b] w3[j] g'(Z2[b][j]), FP32 and as BF16
// hi + lo (the next product's operand).
__global__ void output_grad_kernel(int B, const float* __restrict__ H2,
                                   const float* __restrict__ Z2, const float* __restrict__ w3,
                                   const float* __restrict__ b3, const float* __restrict__ t,
                                   float* __restrict__ dout, float* __restrict__ loss_terms,
                                   float* __restrict__ dZ2, __nv_bfloat16* __restrict__ hi,
                                   __nv_bfloat16* __restrict__ lo) {
  wait_previous();
  const int w = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (w >= B) return;
  const int64_t row = (int64_t)w * kH;
  const float r = output_row(H2 + row, w3, b3[0], lane) - t[w];
  const float d = 2.f * r / (float)B;
  if (lane == 0) {
    dout[w] = d;
    loss_terms[w] = r * r / (float)B;
  }
#pragma unroll
  for (int j = lane; j < kH; j += 32) {
    const float v = d * w3[j] * gelu_grad(Z2[row + j]);
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    dZ2[row + j] = v;
    hi[row + j] = h;
    lo[row + j] = __float2bfloat16_rn(v - __bfloat162float(h));
  }
}

// Mean and standard deviation of l = log(max(fit, 1e-30)) over the batch
// (FP64, fixed order: thread-strided sums then a sequential sum of the 256
// partials).
// Mean and sd of the batch's log-fitness (FP64): 1024 threads, each
// thread's rows summed in order, then a fixed pairwise tree over the
// threads (the same order every run).
__device__ __forceinline__ double tree_sum_1024(double v, double* sh) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  const double t = sh[0];
  __syncthreads();
  return t;
}

// l[b] = log(max(fit[b], 1e-30)) in FP64, over the whole GPU (FP64 is slow
// on one SM)
__global__ void log_fit_kernel(int B, const double* __restrict__ fit, double* __restrict__ l) {
  wait_previous();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const double f = __ldcg(fit + b);
  l[b] = log(f > 1e-30 ? f : 1e-30);
}

__global__ void __launch_bounds__(1024)
target_stats_kernel(int B, const double* __restrict__ l, double* __restrict__ stats) {
  wait_previous();
  __shared__ double sh[1024];
  double a = 0.0;
  for (int b = threadIdx.x; b < B; b += 1024) a += l[b];
  const double mu = tree_sum_1024(a, sh) / B;
  double q = 0.0;
  for (int b = threadIdx.x; b < B; b += 1024) {
    const double d = l[b] - mu;
    q += d * d;
  }
  const double t = tree_sum_1024(q, sh);
  if (threadIdx.x == 0) {
    const double sd = sqrt(t / B);
    stats[0] = mu;
    stats[1] = sd > 0.0 ? sd : 1.0;
  }
}

// The standardised targets t[b] = (l[b] - mean) / sd.
__global__ void targets_kernel(int B, const double* __restrict__ l,
                               const double* __restrict__ stats, float* __restrict__ t) {
  wait_previous();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) t[b] = (float)((l[b] - stats[0]) / stats[1]);
}

// s[j] = sum_b X[b][j] y[b] (y = NULL: plain column sum) over columns j0 ..
// j0 + 31 of [B][256] by 1024 threads: thread (slice, column) adds its slice's
// rows in order, then the 32 slice sums of a column are added in slice order --
// a fixed order, so the result is the same run to run.
constexpr int kColSlices = 32;
__device__ __forceinline__ void colsum_32(int B, int j0, const float* __restrict__ X,
                                          const float* __restrict__ y, float* __restrict__ s) {
  __shared__ float part[kColSlices][33];
  const int c = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int j = j0 + c;
  const int per = (B + kColSlices - 1) / kColSlices;
  const int b0 = sl * per, b1 = min(B, b0 + per);
  float acc = 0.f;
  for (int b = b0; b < b1; b += 16) {   // 16 rows' loads in flight
    float x[16], w[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int bb = b + u < b1 ? b + u : b0;
      x[u] = X[(int64_t)bb * kH + j];
      w[u] = y ? y[bb] : 1.f;
    }
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (b + u < b1) acc = fmaf(x[u], w[u], acc);
  }
  part[sl][c] = acc;
  __syncthreads();
  if (sl == 0) {
    float t = 0.f;
    for (int k = 0; k < kColSlices; ++k) t += part[k][c];
    s[j] = t;
  }
}

// s[0] = sum_b v[b], 256 strided sums added in order, by the first 256 threads.
__device__ __forceinline__ void sum_256(int B, const float* __restrict__ v,
                                        float* __restrict__ s) {
  __shared__ float part[256];
  if (threadIdx.x < 256) {
    float acc = 0.f;
    for (int b = threadIdx.x; b < B; b += 256) acc += v[b];
    part[threadIdx.x] = acc;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int i = 0; i < 256; ++i) t += part[i];
    s[0] = t;
  }
}

// The gradients that are sums over the batch: CTAs 0-7 gw3 = sum_b dout[b]
// H2[b], 8-15 gb2 = sum_b dZ2[b], 16-23 gb1 = sum_b dZ1[b], 24 gb3 = sum_b
// dout[b], 25 the loss.
__global__ void __launch_bounds__(1024)
sums_kernel(int B, const float* __restrict__ H2, const float* __restrict__ dout,
            const float* __restrict__ dZ2, const float* __restrict__ dZ1,
            const float* __restrict__ loss_terms, float* __restrict__ gw3,
            float* __restrict__ gb2, float* __restrict__ gb1, float* __restrict__ gb3,
            float* __restrict__ loss) {
  wait_previous();
  const int what = blockIdx.x / (kH / 32), j0 = (blockIdx.x % (kH / 32)) * 32;
  if (what == 0) colsum_32(B, j0, H2, dout, gw3);
  else if (what == 1) colsum_32(B, j0, dZ2, nullptr, gb2);
  else if (what == 2) colsum_32(B, j0, dZ1, nullptr, gb1);
  else if (j0 == 0) sum_256(B, dout, gb3);
  else sum_256(B, loss_terms, loss);
}

// BF16 copies of one weight: W1b [256][Kq], W2b [256][256] and its transpose.
__device__ __forceinline__ void copy_weight(int64_t e, float w, int K, int Kq,
                                            __nv_bfloat16* __restrict__ W1b,
                                            __nv_bfloat16* __restrict__ W2b,
                                            __nv_bfloat16* __restrict__ W2t) {
  const int64_t n1 = (int64_t)kH * K, w2 = e - n1 - kH;
  const __nv_bfloat16 b = __float2bfloat16_rn(w);
  if (e < n1) {
    const int r = (int)((uint32_t)e / (uint32_t)K);
    W1b[(int64_t)r * Kq + ((int)e - r * K)] = b;
  } else if (w2 >= 0 && w2 < kH * kH) {
    W2b[w2] = b;
    W2t[(w2 % kH) * kH + w2 / kH] = b;
  }
}

__global__ void copy_weights_kernel(int64_t n, int K, int Kq, const float* __restrict__ w,
                                    __nv_bfloat16* __restrict__ W1b,
                                    __nv_bfloat16* __restrict__ W2b,
                                    __nv_bfloat16* __restrict__ W2t) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    copy_weight(e, w[e], K, Kq, W1b, W2b, W2t);
}

// The weight gradients' split sums, in order, into g; then, with apply, Adam and
// the weights' BF16 copies.
__global__ void adam_kernel(int64_t n, int K, int Kq, int splits,
                            const float* __restrict__ parts1, const float* __restrict__ parts2,
                            float* __restrict__ w, float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, bool apply, float lr, float b1, float b2,
                            float eps, float c1, float c2, __nv_bfloat16* __restrict__ W1b,
                            __nv_bfloat16* __restrict__ W2b, __nv_bfloat16* __restrict__ W2t) {
  wait_previous();
  const int64_t n1 = (int64_t)kH * K;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w2 = e - n1 - kH;
    const bool in1 = e < n1, in2 = w2 >= 0 && w2 < kH * kH;
    float gi;
    if (in1 || in2) {
      const float* part = in1 ? parts1 + e : parts2 + w2;
      const int64_t step = in1 ? n1 : (int64_t)kH * kH;
      gi = 0.f;
      for (int z = 0; z < splits; z += 8) {   // eight loads in flight
        float p[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) p[u] = part[(z + u < splits ? z + u : z) * step];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (z + u < splits) gi += p[u];
      }
      g[e] = gi;
    } else {
      gi = g[e];
    }
    if (!apply) continue;
    const float mi = b1 * m[e] + (1.f - b1) * gi;
    const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    const float mh = mi / c1, vh = vi / c2;
    const float wn = w[e] - lr * mh / (sqrtf(vh) + eps);
    w[e] = wn;
    copy_weight(e, wn, K, Kq, W1b, W2b, W2t);
  }
}

__global__ void init_params_kernel(uint64_t seed, int K, float* __restrict__ w) {
  const int64_t n1 = (int64_t)kH * K, n2 = (int64_t)kH * kH;
  const int64_t total = n1 + kH + n2 + kH + kH + 1;
  const float a1 = 1.f / sqrtf((float)K), a2 = 1.f / sqrtf((float)kH);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    int layer;
    int64_t idx;
    float a;
    if (e < n1) {
      layer = 1, idx = e, a = a1;
    } else if (e < n1 + kH) {
      w[e] = 0.f;
      continue;
    } else if (e < n1 + kH + n2) {
      layer = 2, idx = e - n1 - kH, a = a2;
    } else if (e < n1 + kH + n2 + kH) {
      w[e] = 0.f;
      continue;
    } else if (e < n1 + kH + n2 + 2 * kH) {
      layer = 3, idx = e - n1 - 2 * kH - n2, a = a2;
    } else {
      w[e] = 0.f;
      continue;
    }
    const uint32_t r =
        philox4x32_10(seed, (uint32_t)layer, (uint32_t)idx, 0u, kTagSurrogate).x;
    // u in [-1, 1): (r >> 8) 2^-23 - 1, exact in FP32
    const float u = (float)(r >> 8) * (1.0f / 8388608.0f) - 1.0f;
    w[e] = u * a;
  }
}

// ---- screening: keep the n_keep smallest predictions of n ----
constexpr int kScreenThreads = 1024, kScreenWarps = kScreenThreads / 32;

// One CTA. Predictions as order-preserving 32-bit keys in shared memory; four
// 8-bit histogram passes find the n_keep-th smallest key; smaller keys are kept
// and, of the equal ones, the first slots. Each warp then owns a contiguous
// range of slots, so ballots number the kept ones in slot order:
// flag[i] and, for the j-th kept child i, list[j] = i. (A bitonic sort of 16,384 64-bit keys, then a scan, took 206 us.)
__global__ void __launch_bounds__(kScreenThreads)
screen_kernel(int n, int n_keep, const float* __restrict__ pred, int* __restrict__ flag,
              int* __restrict__ list, const int* __restrict__ trusted,
              int* __restrict__ used_trust) {
  wait_previous();
  extern __shared__ uint32_t key[];
  __shared__ int hist[256];
  __shared__ uint32_t prefix;
  __shared__ int want, wless[kScreenWarps], wequal[kScreenWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int trust = *trusted;
  if (tid == 0) *used_trust = trust;
  if (!trust) {   // the exact evaluator stands in: the unscreened generation's children
    for (int i = tid; i < n; i += kScreenThreads) {
      flag[i] = i < n_keep ? 1 : 0;
      if (i < n_keep) list[i] = i;
    }
    return;
  }
  for (int i = tid; i < n; i += kScreenThreads) {
    float p = pred[i];
    if (isnan(p)) p = __int_as_float(0x7f800000);   // NaN ranks last (+inf)
    const uint32_t u = __float_as_uint(p);
    key[i] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);   // float order as unsigned
  }
  if (tid == 0) {
    prefix = 0;
    want = n_keep;   // place of the wanted key among those with the prefix (1-based)
  }
  for (int shift = 24; shift >= 0; shift -= 8) {
    if (tid < 256) hist[tid] = 0;
    __syncthreads();
    const uint32_t pre = prefix;
    for (int i = tid; i < n; i += kScreenThreads) {
      const uint32_t k = key[i];
      if (shift == 24 || (k >> (shift + 8)) == (pre >> (shift + 8)))
        atomicAdd(&hist[(k >> shift) & 255u], 1);
    }
    __syncthreads();
    if (warp == 0) {   // the bin that holds the wanted place
      int h[8], sum = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        h[u] = hist[lane * 8 + u];
        sum += h[u];
      }
      int inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      int before = inc - sum;
      const int w = want;
      __syncwarp();
      if (before < w && w <= inc) {
        int u = 0;
        while (before + h[u] < w) before += h[u++];
        want = w - before;
        prefix = pre | ((uint32_t)(lane * 8 + u) << shift);
      }
    }
    __syncthreads();
  }
  const uint32_t T = prefix;
  const int take = want;   // equal keys to keep
  const int per = (n + kScreenThreads - 1) / kScreenThreads * 32;   // slots per warp
  const int lo = min(n, warp * per), hi = min(n, lo + per);
  int less = 0, equal = 0;
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const bool in = i < hi;
    const uint32_t k = in ? key[i] : 0u;
    less += __popc(__ballot_sync(0xffffffffu, in && k < T));
    equal += __popc(__ballot_sync(0xffffffffu, in && k == T));
  }
  if (lane == 0) {
    wless[warp] = less;
    wequal[warp] = equal;
  }
  __syncthreads();
  int eq = 0, kept = 0;   // equal keys, kept children before this warp's range
  for (int w = 0; w < warp; ++w) {
    kept += wless[w];
    eq += wequal[w];
  }
  kept += min(eq, take);
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const bool in = i < hi;
    const uint32_t k = in ? key[i] : 0u;
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t em = __ballot_sync(0xffffffffu, in && k == T);
    const bool keep = in && (k < T || (k == T && eq + __popc(em & below) < take));
    const uint32_t km = __ballot_sync(0xffffffffu, keep);
    if (in) {
      flag[i] = keep ? 1 : 0;
      if (keep) list[kept + __popc(km & below)] = i;
    }
    eq += __popc(em);
    kept += __popc(km);
  }
}

// next: rows 0..E-1 the elites, row E + j offspring slot E + list[j]; a warp per row.
__global__ void gather_kernel(int rows, int E, int K, const int* __restrict__ list,
                              const float* __restrict__ off, float* __restrict__ next) {
  wait_previous();
  const int r = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (r >= rows) return;
  const int64_t from = r < E ? r : E + list[r - E];
  for (int k = threadIdx.x & 31; k < K; k += 32) next[(int64_t)r * K + k] = off[from * K + k];
}

// Pearson correlation of the kept children's predictions with their exact
// log-fitness, FP64 sums in a fixed order; trusted = r > 0.25. A cluster of 8
// CTAs (FP64 is two operations a cycle and SM): a thread takes every 2048th
// kept child, a warp's sums are exchanged so that lane 4 q ends with sum q, the
// 64 warps' go to the leader's shared memory, six of its threads add them.
constexpr int kTrustCtas = 8, kTrustThreads = 256;
constexpr int kTrustWarps = kTrustCtas * kTrustThreads / 32;
__global__ void __cluster_dims__(kTrustCtas, 1, 1) __launch_bounds__(kTrustThreads)
trust_kernel(int n_kept, const float* __restrict__ pred, const int* __restrict__ list,
             const double* __restrict__ lfit_kept, float* __restrict__ r_out,
             int* __restrict__ trusted) {
  wait_previous();
  __shared__ double sh[kTrustWarps][8];
  __shared__ double tot[8];
  ptx::cluster_arrive();
  const int rank = (int)ptx::cluster_ctarank(), lane = threadIdx.x & 31;
  const int w = rank * (kTrustThreads / 32) + (threadIdx.x >> 5);
  double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int j = rank * kTrustThreads + threadIdx.x; j < n_kept; j += kTrustCtas * kTrustThreads) {
    const double x = pred[list[j]];
    const double y = lfit_kept[j];
    a[0] += 1.0;
    a[1] += x;
    a[2] += y;
    a[3] = fma(x, y, a[3]);
    a[4] = fma(x, x, a[4]);
    a[5] = fma(y, y, a[5]);
  }
  int q0 = 0;
#pragma unroll
  for (int o = 16, m = 4; o >= 4; o >>= 1, m >>= 1) {
    const bool up = (lane & o) != 0;
    q0 += up ? m : 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < m) {
        const double give = up ? a[q] : a[q + m];
        const double keep = up ? a[q + m] : a[q];
        a[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
      }
  }
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 2);
  a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
  ptx::cluster_wait();   // the leader runs
  if ((lane & 3) == 0)
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(
                     ptx::mapa(ptx::smem_addr(&sh[w][q0]), 0)),
                 "d"(a[0])
                 : "memory");
  ptx::cluster_sync();
  if (rank != 0) return;
  if (threadIdx.x < 6) {
    double t[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < kTrustWarps; ++i) t[i & 3] += sh[i][threadIdx.x];
    tot[threadIdx.x] = (t[0] + t[1]) + (t[2] + t[3]);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double* t = tot;
    const double c = t[0];
    double r = 0.0;
    if (c > 1.0) {
      const double cov = t[3] / c - (t[1] / c) * (t[2] / c);
      const double vx = t[4] / c - (t[1] / c) * (t[1] / c);
      const double vy = t[5] / c - (t[2] / c) * (t[2] / c);
      r = (vx > 0.0 && vy > 0.0) ? cov / sqrt(vx * vy) : 0.0;
    }
    *r_out = (float)r;
    *trusted = r > 0.25 ? 1 : 0;
  }
}

// Split-K factor of the weight-gradient GEMMs (reduction over the batch):
// about 64 rows per split, at most kMaxSplits.
int kGradSplits(int B) {
  int sp = (B + 63) / 64;
  return sp < 1 ? 1 : (sp > kMaxSplits ? kMaxSplits : sp);
}

int grid1d(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b < 1) b = 1;
  if (b > 8192) b = 8192;
  return (int)b;
}

template <int NA>
cudaError_t gemm_nt(const NtArgs& a, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(
      gemm_nt_kernel<NA>, cudaFuncAttributeMaxDynamicSharedMemorySize, nt_smem<NA>());
  if (e != cudaSuccess) return e;
  return launch_behind(gemm_nt_kernel<NA>, dim3(kH / kGTN, (a.M + 127) / 128), kGThreads,
                       nt_smem<NA>(), st, a);
}

}  // namespace

int64_t surrogate_param_count(int K) {
  return (int64_t)kH * K + kH + (int64_t)kH * kH + kH + kH + 1;
}

int surrogate_kq(int K) { return (K + kGTK - 1) / kGTK * kGTK; }

cudaError_t surrogate_weights_changed(const SurrogateDev& s, cudaStream_t st) {
  const int64_t n = surrogate_param_count(s.K);
  const int Kq = surrogate_kq(s.K);
  cudaError_t e = cudaMemsetAsync(s.W1b, 0, (size_t)kH * Kq * sizeof(__nv_bfloat16), st);
  if (e != cudaSuccess) return e;
  copy_weights_kernel<<<grid1d(n), 256, 0, st>>>(n, s.K, Kq, s.w, s.W1b, s.W2b, s.W2t);
  return cudaGetLastError();
}

cudaError_t surrogate_init(const SurrogateDev& s, uint64_t seed, cudaStream_t st) {
  const int64_t n = surrogate_param_count(s.K);
  init_params_kernel<<<grid1d(n), 256, 0, st>>>(seed, s.K, s.w);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(s.m, 0, n * sizeof(float), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(s.v, 0, n * sizeof(float), st);
  return e == cudaSuccess ? surrogate_weights_changed(s, st) : e;
}

cudaError_t surrogate_to_bf16(int K, const float* X, int B, __nv_bfloat16* Xb, cudaStream_t st) {
  const int Kq = surrogate_kq(K);
  return launch_behind(to_bf16_kernel, grid1d((int64_t)B * Kq / 8), 256, 0, st, B, K, Kq, X, Xb);
}

cudaError_t surrogate_targets(const SurrogateDev& s, const double* fit, int B, float* t,
                              cudaStream_t st) {
  if (B > s.Bmax) return cudaErrorInvalidValue;
  cudaError_t e = launch_behind(log_fit_kernel, (B + 255) / 256, 256, 0, st, B, fit, s.lfit);
  if (e == cudaSuccess)
    e = launch_behind(target_stats_kernel, 1, 1024, 0, st, B, s.lfit, s.tstat);
  if (e != cudaSuccess) return e;
  return launch_behind(targets_kernel, (B + 255) / 256, 256, 0, st, B, s.lfit, s.tstat, t);
}

namespace {

// Both hidden layers of B rows Xb; keep: Z1, H1, Z2 for a backward pass too.
cudaError_t hidden_layers(const SurrogateDev& s, const __nv_bfloat16* Xb, int B, int keep,
                          cudaStream_t st) {
  const float* b1 = s.w + (int64_t)kH * s.K;
  const float* b2 = b1 + kH + (int64_t)kH * kH;
  NtArgs a{};
  a.M = B;
  a.nkb = surrogate_kq(s.K) / kGTK;
  a.mode = kLayer;
  a.keep = keep;
  a.A = Xb;
  a.B = s.W1b;
  a.bias = b1;
  a.Z = s.Z1;
  a.H = s.H1;
  a.Hb = s.H1b;
  a.status = s.status;
  cudaError_t e = gemm_nt<1>(a, st);   // Z1 = bf(X) bf(W1)^T + b1, H1 = bf(g(Z1))
  if (e != cudaSuccess) return e;
  a.nkb = kH / kGTK;
  a.A = s.H1b;
  a.B = s.W2b;
  a.bias = b2;
  a.Z = s.Z2;
  a.H = s.H2;
  a.Hb = nullptr;
  return gemm_nt<1>(a, st);            // Z2 = H1 bf(W2)^T + b2, H2 = g(Z2)
}

}  // namespace

// Predictions of B rows X [B][K] (FP32 genes) into out [B].
cudaError_t surrogate_forward(const SurrogateDev& s, const float* X, int B, float* out,
                              cudaStream_t st) {
  if (B > s.Bmax) return cudaErrorInvalidValue;
  const float* w3 = s.w + (int64_t)kH * s.K + kH + (int64_t)kH * kH + kH;
  cudaError_t e = surrogate_to_bf16(s.K, X, B, s.Xb, st);
  if (e == cudaSuccess) e = hidden_layers(s, s.Xb, B, 0, st);
  if (e != cudaSuccess) return e;
  return launch_behind(output_kernel, (int)(((int64_t)B * 32 + 255) / 256), 256, 0, st, B, s.H2, w3,
                       w3 + kH, out);
}

// The gradient of the mean squared error over the batch into s.g, the loss into
// s.loss[0]; with apply, an Adam step on it.
cudaError_t surrogate_step(SurrogateDev& s, const SurrogateBatch& bt, bool apply,
                           cudaStream_t st) {
  const int B = bt.n, K = s.K;
  if (B > s.Bmax) return cudaErrorInvalidValue;
  const float* w3 = s.w + (int64_t)kH * K + kH + (int64_t)kH * kH + kH;
  float* gb1 = s.g + (int64_t)kH * K;
  float* gb2 = gb1 + kH + (int64_t)kH * kH;
  float* gw3 = gb2 + kH;
  float* gb3 = gw3 + kH;
  cudaError_t e = hidden_layers(s, bt.Xb, B, 1, st);
  if (e != cudaSuccess) return e;
  e = launch_behind(output_grad_kernel, (int)(((int64_t)B * 32 + 255) / 256), 256, 0, st, B, s.H2,
                    s.Z2, w3, w3 + kH, bt.t, s.dout, s.lterm, s.dZ2, s.dZ2h, s.dZ2l);
  if (e != cudaSuccess) return e;
  // dZ1 = (dZ2 bf(W2)) g'(Z1)
  NtArgs a{};
  a.M = B;
  a.nkb = kH / kGTK;
  a.mode = kDelta;
  a.A = s.dZ2h;
  a.A2 = s.dZ2l;
  a.B = s.W2t;
  a.Zin = s.Z1;
  a.H = s.dZ1;
  a.status = s.status;
  e = gemm_nt<2>(a, st);
  if (e != cudaSuccess) return e;
  // gW1 = dZ1^T bf(X), gW2 = dZ2^T H1, as split sums
  const int splits = kGradSplits(B);
  int kz = (B + splits - 1) / splits;
  kz = (kz + kGTK - 1) / kGTK * kGTK;
  const GradProblem p1{s.dZ1, bt.X, s.split1, K, (K + kGTN - 1) / kGTN};
  const GradProblem p2{s.dZ2, s.H1, s.split2, kH, kH / kGTN};
  constexpr int smem = 2 * (2 * 128 * 128 + kGTN * 128) + 1024 + 64;
  e = cudaFuncSetAttribute(grad_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = launch_behind(grad_gemm_kernel, dim3(p1.tiles + p2.tiles, kH / 128, splits), kGThreads, smem,
                    st, B, p1, p2, kz, s.status);
  if (e == cudaSuccess)
    e = launch_behind(sums_kernel, 3 * (kH / 32) + 2, 1024, 0, st, B, s.H2, s.dout, s.dZ2, s.dZ1,
                      s.lterm, gw3, gb2, gb1, gb3, s.loss);
  if (e != cudaSuccess) return e;
  float c1 = 1.f, c2 = 1.f;
  if (apply) {
    s.step += 1;
    c1 = 1.f - powf(kAdamB1, (float)s.step);
    c2 = 1.f - powf(kAdamB2, (float)s.step);
  }
  const int64_t n = surrogate_param_count(K);
  return launch_behind(adam_kernel, grid1d(n), 256, 0, st, n, K, surrogate_kq(K), splits, s.split1,
                       s.split2, s.w, s.g, s.m, s.v, apply, kAdamLr, kAdamB1, kAdamB2, kAdamEps, c1,
                       c2, s.W1b, s.W2b, s.W2t);
}

cudaError_t surrogate_trust_check(const SurrogateDev& s, int n_kept, const float* pred,
                                  const int* list, const double* fit_kept, float* r_out,
                                  int* trusted, cudaStream_t st) {
  if (n_kept > s.Bmax) return cudaErrorInvalidValue;
  // the kept children's log-fitness over the whole GPU first (FP64)
  const cudaError_t e = launch_behind(log_fit_kernel, (n_kept + 255) / 256, 256, 0, st, n_kept,
                                      fit_kept, s.lfit);
  if (e != cudaSuccess) return e;
  return launch_behind(trust_kernel, kTrustCtas, kTrustThreads, 0, st, n_kept, pred, list, s.lfit,
                       r_out, trusted);
}

cudaError_t surrogate_screen(int n, int n_keep, int E, int K, const float* pred, int* flag,
                             int* list, const float* off, float* next, const int* trusted,
                             int* used_trust, cudaStream_t st) {
  if (n > kScreenMax || n_keep > n || n_keep < 1) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(screen_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(kScreenMax * sizeof(uint32_t)));
  if (e != cudaSuccess) return e;
  e = launch_behind(screen_kernel, 1, kScreenThreads, (size_t)n * sizeof(uint32_t), st, n, n_keep,
                    pred, flag, list, trusted, used_trust);
  if (e != cudaSuccess) return e;
  const int rows = E + n_keep;
  return launch_behind(gather_kernel, (rows * 32 + 255) / 256, 256, 0, st, rows, E, K, list, off,
                       next);
}

}  // namespace game
