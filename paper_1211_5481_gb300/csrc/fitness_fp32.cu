// fitness_fp32.cu -- fitness of a population with the contraction on CUDA-core
// FP32 FFMA (the plain FP32 form).
//
// For chromosome p and pattern m (paper Section 3):
//   Out_p(m) = a_{p,0} + sum_c a_{p,c+1} phi_c(x_m)         (Eq. 2)
//   fit_p    = (1/M) sum_m (y_m - Out_p(m))^2               (Eq. 3, MSE)
// What bounds it: the FP32 FMA pipe (152 SMs x 128 lanes; 5.27e11 flop at
// M = 10^6, P = 1024, K = 257 take 6.6 ms at 2.07 GHz). Register-blocked outer
// products of scalar FMAs reach 54 TFLOP/s on this chip even without memory
// traffic (three register operands per FMA); packed fma.rn.f32x2 ones 70.
// So two chromosomes share one packed FMA: the gene pairs come straight out of
// popT's order, the expansion values are stored in shared memory twice
// (phi, phi), and no register moves build the operands.
//
// A CTA owns 16 U chromosomes and walks pattern tiles of 128 (grid-strided over
// blockIdx.y), in K-chunks of 16 columns through a ring of stages. Warps 0-7
// hold the output block in registers, U x 8 per thread (U = 16: 64 packed FMAs
// per 8 shared loads). Warps 8-11 fill the stages: each thread streams one
// pattern's expansion, its recurrence running on from chunk to chunk (one
// sincosf per feature, the next feature loaded a feature ahead), and one thread
// bulk-copies the chunk's gene rows; so generation and its memory latency run
// beside the FMAs instead of between them. Neither phi nor the output block
// ever reaches global memory: the epilogue forms the residuals, squares them
// (or, for the MAE, takes their absolute values) and sums them over the tile's
// patterns (FP32, 128 terms), and adds the tile sum to an FP64 accumulator per
// chromosome. Each CTA writes its FP64 sums to part[blockIdx.y][p]; the reduce
// kernel adds the rows in a fixed order. Every output's products are added in
// column order and every tile's squares in the same tree for every U, so U
// changes nothing but the FP64 order of the tile sums.
// Measured (U = 16, M = 10^6, N = 32, degree 8, P = 1024): 9.28 ms
// against 11.57 ms with one scalar FMA per product, 8 x 8 outputs per thread
// and generation between the FMAs of the same warps.
#include <type_traits>

#include "basis.cuh"
#include "game_internal.cuh"
#include "tc_common.cuh"
#include "tc_ptx.cuh"

namespace game {

namespace {

using tc::wait_bar;
using tc::wait_bar_drain;

constexpr int BM = 128;   // patterns per tile
constexpr int KC = 16;    // contraction columns per chunk
constexpr int kConsumers = 256, kProducers = 128;
constexpr int kThreads = kConsumers + kProducers;
constexpr int kStages = 4;

template <int U>
struct Fp32Smem {
  float As[kStages][KC][16 * U];   // genes [column][chromosome]
  float2 Bs[kStages][KC][BM];      // (phi, phi) per pattern, in the order b_slot gives
  double sse[16 * U];
  uint64_t a_full[kStages], b_full[kStages], empty[kStages];
  int abort_flag;
};

// Place of pattern p's pair in a row of Bs: the 16 pattern groups of a warp read
// their 16-byte halves (two patterns) from 256 consecutive bytes.
__device__ __forceinline__ int b_slot(int p) {
  return (((p >> 6) * 2 + ((p >> 1) & 1)) * 16 + ((p >> 2) & 15)) * 2 + (p & 1);
}

// The producer role's place in the ring, and one stage's start and end.
struct Producer {
  uint32_t As, Bs;                     // stage 0 of the genes, this thread's pair of stage 0
  uint32_t a_bytes;                    // one stage of genes
  uint32_t a_full, b_full, empty;      // barriers of stage 0
  const float* genes;                  // popT at the CTA's first chromosome
  int Ppad, row_bytes;
  int gp;                              // pattern of the tile
  int stage, uses, issued;             // uses: completed passes over the ring
  volatile int* abort_flag;
  int* status;
  bool ok;
  __device__ __forceinline__ void open(int kc) {   // chunk kc's stage may be filled
    ok = ok && wait_bar(empty + 8u * stage, (uint32_t)(uses & 1) ^ 1u, abort_flag, status);
    if (ok && gp == 0) {
      const uint32_t bar = a_full + 8u * stage;
      ptx::mbar_arrive_expect_tx(bar, (uint32_t)(KC * row_bytes));
      for (int r = 0; r < KC; ++r)
        ptx::bulk_g2s(As + (uint32_t)stage * a_bytes + (uint32_t)(r * row_bytes),
                      genes + (int64_t)(kc * KC + r) * Ppad, (uint32_t)row_bytes, bar);
      ++issued;
    }
  }
  __device__ __forceinline__ void close() {
    if (ok) ptx::mbar_arrive(b_full + 8u * stage);
    if (++stage == kStages) {
      stage = 0;
      ++uses;
    }
  }
  __device__ __forceinline__ void put1(int k, float v) const {   // column k of the open chunk
    asm volatile("st.shared.v2.f32 [%0], {%1, %1};" ::"r"(
                     Bs + (uint32_t)(stage * KC + k) * (BM * 8)),
                 "f"(v)
                 : "memory");
  }
  // 8 columns of the open chunk, its first or second half
  __device__ __forceinline__ void put8(int half, const float (&v)[8]) const {
    const uint32_t at = Bs + (uint32_t)(stage * KC + half * 8) * (BM * 8);
#pragma unroll
    for (int e = 0; e < 8; ++e)
      asm volatile("st.shared.v2.f32 [%0], {%1, %1};" ::"r"(at + (uint32_t)(e * BM * 8)),
                   "f"(v[e])
                   : "memory");
  }
};

// One tile's expansion with the basis and the degree compile-time constants:
// whole features, one FMA per value (the values of basis_run bit for bit),
// stored 8 columns at a time. x: features of the thread's pattern, kPatBlock
// apart; the next group's are loaded while this group's values are formed.
template <int BASIS, int D>
__device__ __noinline__ Producer produce_tile(Producer p, const float* __restrict__ x, int N,
                                              int nch) {
  using FG = FeatureGroup<BASIS, D>;
  float xn[FG::F];
#pragma unroll
  for (int f = 0; f < FG::F; ++f) xn[f] = f < N ? x[f * kPatBlock] : 0.f;
  int u = 0;   // unit (8 columns) to be stored next
  for (int i0 = 0; i0 < N; i0 += FG::F) {
    float xc[FG::F];
#pragma unroll
    for (int f = 0; f < FG::F; ++f) {
      xc[f] = xn[f];
      const int i = i0 + FG::F + f;
      xn[f] = i < N ? x[i * kPatBlock] : 0.f;
    }
    float v[8];
#pragma unroll
    for (int f = 0; f < FG::F; ++f) {
      const bool on = i0 + f < N;
      float fm = 1.f, fv = xc[f], s1 = 0.f;
      if (BASIS == GAME_BASIS_TRIG) {
        float c1;
        sincosf(xc[f], &s1, &c1);
        fv = c1;
      }
      const float c2 = fv + fv;
#pragma unroll
      for (int e = 0; e < FG::W; ++e) {
        if (e > 0) {
          if (BASIS == GAME_BASIS_TRIG && e == D) {
            fm = 0.f;
            fv = s1;
          } else {
            const float fn = fmaf(c2, fv, -fm);
            fm = fv;
            fv = fn;
          }
        }
        const int c = f * FG::W + e;
        v[c & 7] = on ? fv : 0.f;
        if ((c & 7) == 7) {
          if (u < 2 * nch) {   // (units past the last chunk hold no column)
            if ((u & 1) == 0) p.open(u >> 1);
            if (!p.ok) return p;
            p.put8(u & 1, v);
            if (u & 1) p.close();
          }
          ++u;
        }
      }
    }
  }
  const float zero[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (; u < 2 * nch; ++u) {
    if ((u & 1) == 0) p.open(u >> 1);
    if (!p.ok) return p;
    p.put8(u & 1, zero);
    if (u & 1) p.close();
  }
  return p;
}

// Any degree: the same recurrence, straight-line pieces of 8, 4, 2 and 1 columns as
// far as the run of degrees and the chunk go. (With the run's end tested at every
// column this role held narrow CTAs: M = 20,475, P = 128, N = 20, trigonometric degree
// 16: 155 us for 138, N = 24, degree 13: 77 for 73.)
template <int BASIS>
__device__ __noinline__ Producer produce_tile_any(Producer p, const float* __restrict__ x, int N,
                                                  int d, int nch) {
  int i = 0, left = d;   // feature, columns left in its run of degrees
  bool sine = false;     // trigonometric: the sine group
  float f, fm, c2, s1 = 0.f;   // the next column's value, the one before it
  float xn = x[0];
  auto start = [&]() {
    const float xi = xn;
    xn = i + 1 < N ? x[(i + 1) * kPatBlock] : 0.f;
    f = xi;
    if (BASIS == GAME_BASIS_TRIG) sincosf(xi, &s1, &f);
    c2 = f + f;
    fm = 1.f;
  };
  auto run = [&](auto len, int& k) {   // len columns from column k of the open chunk
#pragma unroll
    for (int e = 0; e < decltype(len)::value; ++e) {
      p.put1(k + e, f);
      const float fn = fmaf(c2, f, -fm);
      fm = f;
      f = fn;
    }
    k += decltype(len)::value;
  };
  start();
  for (int kc = 0; kc < nch; ++kc) {
    p.open(kc);
    if (!p.ok) return p;
    int k = 0;
    do {
      int n = min(left, KC - k);
      left -= n;
#pragma unroll 1
      for (; n >= 8; n -= 8) run(std::integral_constant<int, 8>{}, k);
      if (n & 4) run(std::integral_constant<int, 4>{}, k);
      if (n & 2) run(std::integral_constant<int, 2>{}, k);
      if (n & 1) run(std::integral_constant<int, 1>{}, k);
      if (left == 0) {
        left = d;
        if (BASIS == GAME_BASIS_TRIG && !sine) {
          sine = true;
          fm = 0.f;
          f = s1;
        } else {
          sine = false;
          if (++i < N) {
            start();
          } else {   // columns past the last feature's are zero
            f = fm = c2 = 0.f;
            left = nch * KC;
          }
        }
      }
    } while (k < KC);
    p.close();
  }
  return p;
}

__device__ __forceinline__ Producer produce(const Producer& p, const float* x, int N, int d,
                                            int basis, int nch) {
#define GAME_PRODUCE_CASE(D)                                                         \
  case D:                                                                            \
    return basis == GAME_BASIS_CHEB ? produce_tile<GAME_BASIS_CHEB, D>(p, x, N, nch) \
                                    : produce_tile<GAME_BASIS_TRIG, D>(p, x, N, nch);
  switch (d) {
    GAME_PRODUCE_CASE(1)
    GAME_PRODUCE_CASE(2)
    GAME_PRODUCE_CASE(3)
    GAME_PRODUCE_CASE(4)
    GAME_PRODUCE_CASE(5)
    GAME_PRODUCE_CASE(6)
    GAME_PRODUCE_CASE(7)
    GAME_PRODUCE_CASE(8)
    GAME_PRODUCE_CASE(9)
    GAME_PRODUCE_CASE(10)
    default:
      return basis == GAME_BASIS_CHEB ? produce_tile_any<GAME_BASIS_CHEB>(p, x, N, d, nch)
                                      : produce_tile_any<GAME_BASIS_TRIG>(p, x, N, d, nch);
  }
#undef GAME_PRODUCE_CASE
}

template <int U, bool ABS>
__global__ void __launch_bounds__(kThreads, U >= 8 ? 1 : 2)
fitness_fp32_kernel(int64_t M, int N, int d, int basis, int Kc,
                    const float* __restrict__ Xt,
                    const float* __restrict__ y, const float* __restrict__ popT,
                    const float* __restrict__ a0, int Ppad, int ntiles,
                    double* __restrict__ part, int* status) {
  constexpr int BP = 16 * U;              // chromosomes per CTA
  constexpr int NG = U / 4;               // a thread's groups of 4 chromosomes, 64 apart
  extern __shared__ __align__(16) uint8_t smem[];
  wait_previous();
  Fp32Smem<U>& sm = *reinterpret_cast<Fp32Smem<U>*>(smem);
  volatile int* abort_flag = &sm.abort_flag;

  const int tid = threadIdx.x;
  const int cb = blockIdx.x * BP;
  const int nch = Kc / KC;
  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(ptx::smem_addr(&sm.a_full[s]), 1);
      ptx::mbar_init(ptx::smem_addr(&sm.b_full[s]), kProducers);
      ptx::mbar_init(ptx::smem_addr(&sm.empty[s]), kConsumers / 32);
    }
    sm.abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
  }
  for (int i = tid; i < BP; i += kThreads) sm.sse[i] = 0.0;
  __syncthreads();

  if (tid >= kConsumers) {
    // ---------------- producers: expansion and genes ----------------
    if (U == 16) asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    Producer p;
    p.gp = tid - kConsumers;
    p.As = ptx::smem_addr(&sm.As[0][0][0]);
    p.Bs = ptx::smem_addr(&sm.Bs[0][0][b_slot(p.gp)]);
    p.a_bytes = KC * BP * 4;
    p.a_full = ptx::smem_addr(sm.a_full);
    p.b_full = ptx::smem_addr(sm.b_full);
    p.empty = ptx::smem_addr(sm.empty);
    p.genes = popT + cb;
    p.Ppad = Ppad;
    p.row_bytes = BP * 4;
    p.stage = p.uses = p.issued = 0;
    p.abort_flag = abort_flag;
    p.status = status;
    p.ok = true;
    for (int t = blockIdx.y; t < ntiles && p.ok; t += gridDim.y)
      p = produce(p, Xt + (int64_t)t * N * kPatBlock + p.gp, N, d, basis, nch);
    // own copies in flight: the last phase armed on each stage
    if (p.gp == 0)
      for (int s = 0; s < kStages && s < p.issued; ++s)
        wait_bar_drain(p.a_full + 8u * s,
                       (uint32_t)((p.issued - s + kStages - 1) / kStages - 1) & 1u, status);
  } else {
    // ---------------- consumers: products and epilogue ----------------
    if (U == 16) asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    const int tx = tid & 15;   // pattern group
    const int ty = tid >> 4;   // chromosome group
    int stage = 0;
    uint32_t par = 0;
    bool ok = true;
    for (int t = blockIdx.y; t < ntiles && ok; t += gridDim.y) {
      uint64_t acc[U / 2][8];   // chromosome pairs x patterns
#pragma unroll
      for (int u = 0; u < U / 2; ++u)
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[u][v] = 0;

      for (int kc = 0; kc < nch; ++kc) {
        ok = wait_bar(ptx::smem_addr(&sm.a_full[stage]), par, abort_flag, status) &&
             wait_bar(ptx::smem_addr(&sm.b_full[stage]), par, abort_flag, status);
        ok = __all_sync(0xffffffffu, ok);   // a warp leaves as one
        if (!ok) break;
        const float* as = &sm.As[stage][0][ty * 4];
        const ulonglong2* bs = reinterpret_cast<const ulonglong2*>(&sm.Bs[stage][0][0]) + tx;
#pragma unroll
        for (int k = 0; k < KC; ++k) {
          uint64_t a[U / 2], b[8];
#pragma unroll
          for (int g = 0; g < NG; ++g) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(as + k * BP + g * 64);
            a[2 * g] = w.x;
            a[2 * g + 1] = w.y;
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const ulonglong2 w = bs[k * (BM / 2) + j * 16];
            b[2 * j] = w.x;
            b[2 * j + 1] = w.y;
          }
#pragma unroll
          for (int u = 0; u < U / 2; ++u)
#pragma unroll
            for (int v = 0; v < 8; ++v) acc[u][v] = ptx::f2_fma(a[u], b[v], acc[u][v]);
        }
        __syncwarp();
        if ((tid & 31) == 0) ptx::mbar_arrive(ptx::smem_addr(&sm.empty[stage]));
        if (++stage == kStages) {
          stage = 0;
          par ^= 1u;
        }
      }
      if (!ok) break;

      // squared residuals of this thread's outputs; patterns 4 tx + (0..3),
      // then 64 + 4 tx + (0..3), then the 16 pattern groups
      const int64_t mbase = (int64_t)t * BM;
      const float4 y_lo = *reinterpret_cast<const float4*>(y + mbase + tx * 4);
      const float4 y_hi = *reinterpret_cast<const float4*>(y + mbase + 64 + tx * 4);
      const float yv[8] = {y_lo.x, y_lo.y, y_lo.z, y_lo.w, y_hi.x, y_hi.y, y_hi.z, y_hi.w};
      bool in[8];
#pragma unroll
      for (int v = 0; v < 8; ++v) in[v] = mbase + (v < 4 ? tx * 4 + v : 60 + tx * 4 + v) < M;
      float mine = 0.f;   // lane tx keeps chromosome u = tx: one FP64 add per thread
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int cl = (u / 4) * 64 + ty * 4 + u % 4;
        const float bias = a0[cb + cl];
        float s = 0.f;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          const float2 o = ptx::f2_unpack(acc[u / 2][v]);
          const float r = (yv[v] - bias) - ((u & 1) ? o.y : o.x);
          s = in[v] ? (ABS ? s + fabsf(r) : fmaf(r, r, s)) : s;
        }
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 4);
        s += __shfl_xor_sync(0xffffffffu, s, 8);
        if (tx == u) mine = s;
      }
      if (tx < U) sm.sse[(tx / 4) * 64 + ty * 4 + tx % 4] += (double)mine;
    }
  }
  __syncthreads();
  for (int i = tid; i < BP; i += kThreads)
    part[(int64_t)blockIdx.y * Ppad + cb + i] = sm.sse[i];
}

// Resident CTAs per SM of each width (registers).
constexpr int fp32_resident(int U) { return U >= 8 ? 1 : 2; }

}  // namespace

Fp32Plan plan_fp32(const Shape& s, int P, int num_sms) {
  Fp32Plan pl;
  pl.BM = BM;
  pl.Kc = ceil_div(s.Kp, KC) * KC;
  pl.grid_x = ceil_div(P, 128);
  const int ntiles = ceil_div(s.M, BM);
  // The width with the least time: rounds of tiles per CTA x a tile's time.
  // A 16-column chunk of a tile measured 2.85, 1.64 and (two CTAs sharing an
  // SM) 2.6 us for U = 16, 8 and 4; alone on its SM a U = 4 CTA is held by its
  // expansion. Both sides: M = 10^6, K = 257, P = 1024: 9.4 / 10.8 / 17.1 ms
  // (U = 16, 8, 4); P = 64: 2.37 / 1.40 / 1.09 ms; M = 1000, K = 1281,
  // P = 2048: 233 / 135 / 213 us. (U = 2 was never faster than U = 4.)
  double best = 0.0;
  for (int U = 16; U >= 4; U >>= 1) {
    const int gx = ceil_div(P, 16 * U);
    const int slots = fp32_resident(U) * num_sms;
    int gy = slots / gx;
    if (gy < 1) gy = 1;
    if (gy > ntiles) gy = ntiles;
    const int64_t ctas = (int64_t)gx * gy;
    const double tile = U == 16 ? 2.85 : U == 8 ? 1.64 : ctas > num_sms ? 2.6 : 1.5;
    const double cost = (double)ceil_div(ctas, slots) * ceil_div(ntiles, gy) * tile;
    if (U == 16 || cost < best) {
      best = cost;
      pl.U = U;
      pl.cta_x = gx;
      pl.grid_y = gy;
    }
  }
  pl.Ppad = ceil_div((int64_t)pl.cta_x * 16 * pl.U, 128) * 128;
  return pl;
}

cudaError_t launch_fitness_fp32(const Fp32Plan& pl, const Shape& s, const float* Xt,
                                const float* y, const float* popT, const float* a0, int P,
                                int Ppad, double* part, int* status, int err, cudaStream_t st) {
  if (Ppad < pl.Ppad || P > pl.cta_x * 16 * pl.U) return cudaErrorInvalidValue;
  const int ntiles = ceil_div(s.M, BM);
  dim3 grid(pl.cta_x, pl.grid_y);
  auto go = [&](auto kern, int smem) -> cudaError_t {
    const cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    return launch_behind(kern, grid, kThreads, smem, st, s.M, s.N, s.d, s.basis, pl.Kc, Xt, y, popT,
                         a0, Ppad, ntiles, part, status);
  };
  const bool abs = err == GAME_ERR_MAE;
  switch (pl.U) {
    case 16:
      return go(abs ? fitness_fp32_kernel<16, true> : fitness_fp32_kernel<16, false>,
                (int)sizeof(Fp32Smem<16>));
    case 8:
      return go(abs ? fitness_fp32_kernel<8, true> : fitness_fp32_kernel<8, false>,
                (int)sizeof(Fp32Smem<8>));
    case 4:
      return go(abs ? fitness_fp32_kernel<4, true> : fitness_fp32_kernel<4, false>,
                (int)sizeof(Fp32Smem<4>));
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace game
