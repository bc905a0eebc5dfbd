// fitness_tc2.cu -- the BF16 fitness contraction on pairs of SMs
// (tcgen05 cta_group::2), the squared- or absolute-error reduction fused into
// the epilogue.
//
// Math (paper Section 3): Out_p(m) = a_{p,0} + sum_c a_{p,c+1} phi_c(x_m)
// (Eq. 2), fit_p = (1/M) sum_m (y_m - Out_p(m))^2 (Eq. 3, MSE). For a tile of
// 256 patterns the sum over c is the dense product D[p][m] = A[p][:] . PHI[m][:].
//
// A cluster of two CTAs (one per SM of a pair) computes D for 256 chromosomes
// (MMA-M, 128 per CTA: the rows of each CTA's tensor memory) x 256 patterns
// (MMA-N) with one tcgen05.mma.cta_group::2 per K = 16 step, issued by one
// thread of the even CTA: each CTA holds in its shared memory the genes of
// its 128 chromosomes and the expansion of its 128 patterns (half of B), so
// per MMA each SM reads half the operand bytes of a one-SM 128 x 256 MMA,
// and each SM expands only its own 128 patterns of a tile.
//
// Warp roles in each CTA (16 warps):
//   warp 0       gene producer: bulk copies of this CTA's 16 KB gene blocks
//                (chromosome tile 2c + rank, K-block kb) into a ring of stages.
//   warp 1       even CTA: MMA issuer (one thread); both CTAs: tensor-memory
//                allocation of the pair (512 columns: two accumulators of 256).
//   warp 2       feature producer (staged features only): this CTA's
//                128-pattern feature block of the next tile.
//   warp 3       odd CTA: relays the completion of its gene copies to the even
//                CTA's stage barrier (the copy's own barrier is local).
//   warps 4-11   epilogue: tcgen05.ld of this CTA's 128 accumulator rows
//                (warps 4-7 the first 128 pattern columns, 8-11 the second),
//                r = (y_m - a_0) - D, sse += r^2 in packed FP32 pairs, FP64
//                partials per (cluster, column half).
//   warps 12-19  expansion of this CTA's 128 patterns (degrees 1..10 whole
//                features at a time, expand_stream.cuh; beyond, per 8-column
//                chunk): the basis recurrence in registers, BF16, stored in the
//                K-major SWIZZLE_128B layout, into a ring of K-block slots.
// Barriers: the MMA issuer waits on the even CTA's barriers only; the odd
// CTA's producers reach them by cluster-scope arrivals (one per warp for the
// expansion and the epilogue, one relay per gene stage); every MMA commit is
// multicast to the same barrier in both CTAs, so each CTA's producers and
// epilogue wait on their own copies. All waits are bounded (4e9 cycles): on expiry a
// CTA raises the status word, abandons its loops, drains its own copies (the
// even CTA its MMAs), and both CTAs meet at the final cluster barrier before
// the pair's tensor memory is freed.
#include <type_traits>

#include "basis.cuh"
#include "expand_stream.cuh"
#include "game_internal.cuh"
#include "tc_common.cuh"
#include "tc_ptx.cuh"

namespace game {

namespace {

using namespace tc;

constexpr uint32_t kABytes = 128 * 128;   // one CTA's gene block: 128 chromosomes x 64 genes
constexpr int kEpiWarp0 = 4;
constexpr int kBasisWarp0 = 12;
// (eight expansion warps, one elected issuing thread, epilogue one step ahead: M =
// 4 10^6, N = 48, degree 6, P = 2048: 3.02 -> 2.61 ms; M = 94,601, N = 26,
// trigonometric degree 11, P = 1092, the chunk generator: 360 -> 232 us)
constexpr int kBasisThreads = 256;        // warps 12..19
constexpr int kThreads = kBasisWarp0 * 32 + kBasisThreads;
constexpr int kRows = 128;                // patterns of a tile held by one CTA
constexpr int kBN = 2 * kRows;            // patterns per tile (MMA N)
constexpr int kMaxSmem = 232448;          // 227 KB opt-in per CTA
constexpr int kMinSmem = 120 * 1024;      // one CTA per SM
constexpr uint32_t kPhiArrivals = 16;     // expansion warps of both CTAs
constexpr uint32_t kAccArrivals = 16;     // epilogue warps of both CTAs

struct Tc2Args {
  int64_t M;
  int N, d, basis, Kp;
  int KB, Cp, NS, stages, nmma_last, ntiles, Ppad, xstage;
  int ycopy;   // targets of each tile in a two-slot shared buffer
  const float* Xt;
  const float* y;
  const uint8_t* popA;
  const float* a0;
  double* part;
  int* status;
  uint64_t stall_ns;   // test hook (see fitness_tc.cu)
};

struct Smem2 {
  int phi, ast, xs, ys, tab, bars, total;
};

__host__ __device__ inline int num_bars2(int NS, int S) { return 2 * S + 2 * NS + 11; }

__host__ __device__ inline Smem2 smem_plan2(int KB, int NS, int N, int S, int xstage, int ycopy) {
  Smem2 s;
  s.phi = 0;
  s.ast = NS * kRows * 128;
  s.xs = s.ast + S * (int)kABytes;
  s.ys = s.xs + (xstage ? N * kRows * 4 : 0);
  s.tab = s.ys + (ycopy ? 2 * kBN * 4 : 0);
  s.bars = (s.tab + KB * 8 * 4 + 7) & ~7;
  s.total = s.bars + num_bars2(NS, S) * 8 + 16 + 1024;   // + alignment slack
  return s;
}

// The 8 expansion values of chunk `desc` for one pattern whose features are
// xrow[i * xstride] (staged features, degrees above 10): the same values as
// gen_chunk, with the Chebyshev run of one feature's degrees and the crossing
// chunks of d >= 4 on their branch-free generators.
__device__ __forceinline__ void gen8(uint32_t desc, int basis, int d, int N, const float* xrow,
                                     int xstride, float (&v)[8]) {
  if (basis == GAME_BASIS_CHEB && (desc & kChunkRun) && chunk_columns(desc) == 8) {
    const int i = chunk_feature(desc);
    const int j0 = chunk_degree(desc);
    const float x = xrow[i * xstride];
    const float x2 = x + x;
    float t = x, tm = 1.f;
    for (int st = 1; st < j0; ++st) {
      const float n = fmaf(x2, t, -tm);
      tm = t;
      t = n;
    }
    v[0] = t;
#pragma unroll
    for (int e = 1; e < 8; ++e) {
      const float n = fmaf(x2, t, -tm);
      tm = t;
      t = n;
      v[e] = t;
    }
  } else if (basis == GAME_BASIS_CHEB && d >= 4 && !(desc & kChunkZero)) {
    cheb_cross1(desc, d, N, xrow, xstride, v);
  } else {
    gen_chunk(desc, basis, d, N, xrow, xstride, v);
  }
}

__device__ __forceinline__ void store_bf16x8(uint8_t* phik, int r, int qd, const float (&v)[8]) {
  *reinterpret_cast<uint4*>(phik + r * 128 + ((qd ^ (r & 7)) << 4)) =
      make_uint4(bf16x2_bits(v[0], v[1]), bf16x2_bits(v[2], v[3]), bf16x2_bits(v[4], v[5]),
                 bf16x2_bits(v[6], v[7]));
}

// Two Chebyshev runs of 8 degrees (chunks of the features xa and xb, first
// degrees ja and jb), interleaved: two independent recurrences.
__device__ __forceinline__ void cheb_run_pair(float xa, int ja, float xb, int jb, float (&va)[8],
                                              float (&vb)[8]) {
  const float a2 = xa + xa, b2 = xb + xb;
  float ta = xa, tam = 1.f, tb = xb, tbm = 1.f;
  for (int st = 1; st < ja; ++st) {
    const float n = fmaf(a2, ta, -tam);
    tam = ta;
    ta = n;
  }
  for (int st = 1; st < jb; ++st) {
    const float n = fmaf(b2, tb, -tbm);
    tbm = tb;
    tb = n;
  }
  va[0] = ta;
  vb[0] = tb;
#pragma unroll
  for (int e = 1; e < 8; ++e) {
    const float na = fmaf(a2, ta, -tam), nb = fmaf(b2, tb, -tbm);
    tam = ta;
    ta = na;
    tbm = tb;
    tb = nb;
    va[e] = ta;
    vb[e] = tb;
  }
}

template <bool ABS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    fitness_tc2_kernel(const Tc2Args a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int KB = a.KB, N = a.N, S = a.stages, NS = a.NS;
  const Smem2 sp = smem_plan2(KB, NS, N, S, a.xstage, a.ycopy);
  uint8_t* phi = base + sp.phi;
  uint8_t* ast = base + sp.ast;
  float* xs = reinterpret_cast<float*>(base + sp.xs);
  float* ys = reinterpret_cast<float*>(base + sp.ys);
  uint32_t* tab = reinterpret_cast<uint32_t*>(base + sp.tab);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + sp.bars);
  uint64_t* a_full = bars;
  uint64_t* a_empty = a_full + S;
  uint64_t* phi_full = a_empty + S;
  uint64_t* phi_free = phi_full + NS;
  uint64_t* acc_full = phi_free + NS;
  uint64_t* acc_empty = acc_full + 2;
  uint64_t* x_full = acc_empty + 2;
  uint64_t* x_empty = x_full + 1;
  uint64_t* drain = x_empty + 1;
  uint64_t* y_full = drain + 1;    // [2]
  uint64_t* y_empty = y_full + 2;  // [2]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(y_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

  const uint32_t rank = ptx::cluster_ctarank();
  const bool lead = rank == 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      // the even CTA's stage completes on its own copy and the odd CTA's relay
      ptx::mbar_init(ptx::smem_addr(&a_full[s]), lead ? 2 : 1);
      ptx::mbar_init(ptx::smem_addr(&a_empty[s]), 1);
    }
    for (int sl = 0; sl < NS; ++sl) {
      // (features from L2: a K-block is one warpgroup's in each CTA)
      ptx::mbar_init(ptx::smem_addr(&phi_full[sl]), a.xstage ? kPhiArrivals : kPhiArrivals / 2);
      ptx::mbar_init(ptx::smem_addr(&phi_free[sl]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_addr(&acc_full[b]), 1);
      ptx::mbar_init(ptx::smem_addr(&acc_empty[b]), kAccArrivals);
    }
    ptx::mbar_init(ptx::smem_addr(x_full), 1);
    ptx::mbar_init(ptx::smem_addr(x_empty), kBasisThreads);
    ptx::mbar_init(ptx::smem_addr(drain), 1);
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(ptx::smem_addr(&y_full[b]), 1);
      ptx::mbar_init(ptx::smem_addr(&y_empty[b]), kBasisWarp0 - kEpiWarp0);   // epilogue warps
    }
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::fence_proxy_async_smem();
  }
  if (warp == 1) {
    ptx::tmem_alloc2(ptx::smem_addr(tmem_holder), 512u);
    ptx::tmem_relinquish2();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();   // the peer's barriers exist before any arrival on them
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_holder;
  wait_previous();   // (only shared and tensor memory so far)

  const int ncl = (int)(gridDim.x >> 1), cl = (int)(blockIdx.x >> 1);
  const int my_tiles = (a.ntiles - cl + ncl - 1) / ncl;
  const int Cp = a.Cp;

  // each tile's targets into slot it & 1, released by the CTA's epilogue warps
  // after the tile's last chromosome tile: one thread of an otherwise idle warp
  // (the even CTA's relay warp, the odd CTA's issuer warp)
  auto produce_targets = [&]() {
    int issued = 0;
    for (int it = 0; it < my_tiles; ++it) {
      const int b = it & 1;
      if (!wait_bar(ptx::smem_addr(&y_empty[b]), ((it >> 1) & 1) ^ 1, abort_flag, a.status)) break;
      ptx::mbar_arrive_expect_tx(ptx::smem_addr(&y_full[b]), kBN * 4);
      ptx::bulk_g2s(ptx::smem_addr(ys + b * kBN), a.y + ((int64_t)cl + (int64_t)it * ncl) * kBN,
                    kBN * 4, ptx::smem_addr(&y_full[b]));
      ++issued;
    }
    for (int b = 0; b < 2 && b < issued; ++b) {
      const int uses = (issued - b + 1) / 2;
      wait_bar_drain(ptx::smem_addr(&y_full[b]), (uint32_t)(uses - 1) & 1u, a.status);
    }
  };

  // (registers: see fitness_tc.cu)
  if (warp < kEpiWarp0) ptx::regs_dec<80>();
  if (warp == 0) {
    // ---------------- gene producer (both CTAs) ----------------
    if (lane == 0) {
      uint32_t q = 0, s = 0, ph = 0;
      bool ok = true;
      for (int it = 0; it < my_tiles && ok; ++it)
        for (int c = 0; c < Cp && ok; ++c)
          for (int kb = 0; kb < KB && ok; ++kb) {
            ok = wait_bar(ptx::smem_addr(&a_empty[s]), ph ^ 1, abort_flag, a.status);
            if (!ok) break;
            ptx::mbar_arrive_expect_tx(ptx::smem_addr(&a_full[s]), kABytes);
            ptx::bulk_g2s(ptx::smem_addr(ast + s * kABytes),
                          a.popA + ((size_t)(2 * c + (int)rank) * KB + kb) * kABytes, kABytes,
                          ptx::smem_addr(&a_full[s]));
            ++q;
            if (++s == (uint32_t)S) {
              s = 0;
              ph ^= 1;
            }
          }
      // own copies in flight: the last phase armed on each stage
      for (uint32_t st = 0; st < (uint32_t)S && st < q; ++st) {
        const uint32_t uses = (q - st + S - 1) / S;
        wait_bar_drain(ptx::smem_addr(&a_full[st]), (uses - 1) & 1, a.status);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (even CTA) ----------------
    // (one elected thread, running descriptors: see fitness_tc.cu)
    if (lead) {
      const uint32_t idesc = ptx::idesc_bf16_f32(2 * kRows, kBN);
      const uint64_t adesc0 = ptx::desc_kmajor_sw128(ptx::smem_addr(ast));
      const uint64_t bdesc0 = ptx::desc_kmajor_sw128(ptx::smem_addr(phi));
      const uint32_t dhi = (uint32_t)(adesc0 >> 32);
      const uint32_t alo0 = (uint32_t)adesc0, blo0 = (uint32_t)bdesc0;
      const uint32_t a_step = kABytes >> 4;
      const uint32_t b_step = (uint32_t)(kRows * 128) >> 4;
      const uint32_t alo_end = alo0 + (uint32_t)S * a_step, blo_end = blo0 + (uint32_t)NS * b_step;
      const uint32_t a_full0 = ptx::smem_addr(a_full), phi_full0 = ptx::smem_addr(phi_full);
      const uint32_t a_empty_off = 8u * (uint32_t)S, phi_free_off = 8u * (uint32_t)NS;
      const uint32_t acc_full0 = ptx::smem_addr(acc_full), acc_empty0 = ptx::smem_addr(acc_empty);
      const uint16_t both = 3;
      const int nlast = a.nmma_last;
      bool ok = true;
      if (a.stall_ns) {
        // test hook: the drain barrier's first phase completes only at the
        // final commit below, so this wait runs out
        const uint64_t t0 = ptx::global_timer_ns();
        while (ok && !ptx::mbar_try_wait_sleep(ptx::smem_addr(drain), 0, kSuspendNs)) {
          if (ptx::global_timer_ns() - t0 > a.stall_ns) {
            *abort_flag = 1;
            atomicExch(a.status, (int)kDevTimeout);
            ok = false;
          }
        }
        __syncwarp();
        ok = __all_sync(0xffffffffu, ok);
      }
      auto kstep = [&](uint32_t d_tmem, uint32_t al, uint32_t bl, uint32_t acc) {
        ptx::mma_bf16_pair(d_tmem, ((uint64_t)dhi << 32) | al, ((uint64_t)dhi << 32) | bl,
                             idesc, acc);
      };
      if (ptx::elect_one()) {
        uint32_t alo = alo0, abar = a_full0, ph = 0;
        uint32_t tile_blo = blo0, tile_pbar = phi_full0, tile_par = 0;
        uint32_t acc_it = 0;
        for (int it = 0; it < my_tiles && ok; ++it) {
          uint32_t blo = tile_blo, pbar = tile_pbar, par = tile_par;
          for (int c = 0; c < Cp && ok; ++c) {
            const uint32_t buf = acc_it & 1;
            ok = wait_bar(acc_empty0 + 8 * buf, ((acc_it >> 1) & 1) ^ 1, abort_flag, a.status);
            if (!ok) break;
            ptx::tc_fence_after();
            const uint32_t d_tmem = tmem + buf * (uint32_t)kBN;
            blo = tile_blo;
            pbar = tile_pbar;
            par = tile_par;
            for (int kb = 0; kb < KB; ++kb) {
              if (c == 0) {
                ok = wait_bar(pbar, par, abort_flag, a.status);
                if (!ok) break;
              }
              ok = wait_bar(abar, ph, abort_flag, a.status);
              if (!ok) break;
              const int nm = kb == KB - 1 ? nlast : 4;
              kstep(d_tmem, alo, blo, kb != 0);
              if (nm == 4) {
                kstep(d_tmem, alo + 2u, blo + 2u, 1u);
                kstep(d_tmem, alo + 4u, blo + 4u, 1u);
                kstep(d_tmem, alo + 6u, blo + 6u, 1u);
              } else {
                for (int kk = 1; kk < nm; ++kk)
                  kstep(d_tmem, alo + 2u * kk, blo + 2u * kk, 1u);
              }
              ptx::mma_commit_pair_mc(abar + a_empty_off, both);
              if (c == Cp - 1) ptx::mma_commit_pair_mc(pbar + phi_free_off, both);
              if (kb == KB - 1) ptx::mma_commit_pair_mc(acc_full0 + 8 * buf, both);
              alo += a_step;
              abar += 8;
              if (alo == alo_end) {
                alo = alo0;
                abar = a_full0;
                ph ^= 1;
              }
              blo += b_step;
              pbar += 8;
              if (blo == blo_end) {
                blo = blo0;
                pbar = phi_full0;
                par ^= 1u;
              }
            }
            ++acc_it;
          }
          tile_blo = blo;
          tile_pbar = pbar;
          tile_par = par;
        }
        // every MMA issued above has completed once this arrives
        ptx::mma_commit_pair(ptx::smem_addr(drain));
      }
      __syncwarp();
      wait_bar_drain(ptx::smem_addr(drain), 0, a.status);
    } else if (lane == 0 && a.ycopy) {
      produce_targets();
    }
  } else if (warp == 2) {
    // ---------------- feature producer (staged features only) ----------------
    if (lane == 0 && a.xstage) {
      int issued = 0;
      const uint32_t bytes = (uint32_t)(N * kRows * 4);
      for (int it = 0; it < my_tiles; ++it) {
        const int64_t t = (int64_t)cl + (int64_t)it * ncl;
        if (!wait_bar(ptx::smem_addr(x_empty), (it & 1) ^ 1, abort_flag, a.status)) break;
        ptx::mbar_arrive_expect_tx(ptx::smem_addr(x_full), bytes);
        const int64_t blk = t * 2 + rank;   // this CTA's 128-pattern block
        ptx::bulk_g2s(ptx::smem_addr(xs), a.Xt + blk * N * kPatBlock, bytes,
                      ptx::smem_addr(x_full));
        if (it + 1 < my_tiles)
          ptx::bulk_prefetch_l2(a.Xt + ((t + ncl) * 2 + rank) * N * kPatBlock, bytes);
        ++issued;
      }
      if (issued > 0) wait_bar_drain(ptx::smem_addr(x_full), (issued - 1) & 1, a.status);
    }
  } else if (warp == 3) {
    // ---------------- odd CTA: relay of gene-copy completions ----------------
    if (lane == 0 && !lead) {
      const int total = my_tiles * Cp * KB;
      uint32_t s = 0, ph = 0;
      int done = 0;
      for (; done < total; ++done) {
        if (!wait_bar(ptx::smem_addr(&a_full[s]), ph, abort_flag, a.status)) break;
        ptx::mbar_arrive_cluster(ptx::mapa(ptx::smem_addr(&a_full[s]), 0));
        if (++s == (uint32_t)S) {
          s = 0;
          ph ^= 1;
        }
      }
    } else if (lane == 0 && a.ycopy) {
      produce_targets();
    }
  } else if (warp >= kEpiWarp0 && warp < kBasisWarp0) {
    // ---------------- epilogue (both CTAs) ----------------
    const int qw = warp & 3;
    ptx::regs_inc<104>();
    const int half = (warp - kEpiWarp0) >> 2;
    const int row = qw * 32 + lane;
    const int col_lo = half * kRows;
    const uint32_t lane_addr = (uint32_t)(qw * 32) << 16;
    double* part_row = a.part + (size_t)(2 * cl + half) * a.Ppad;
    const uint32_t acc_empty_lead0 = ptx::mapa(ptx::smem_addr(acc_empty), 0);
    // (what bounds it: see epi_reduce's header)
    auto reduce_tiles = [&](auto ys_tag) {
      constexpr bool YS = decltype(ys_tag)::value;
      uint32_t acc_it = 0;
      bool ok = true;
      LastSum last;
      float bias_n = a.a0[(int)rank * kRows + row];   // the next accumulator's
      for (int it = 0; it < my_tiles && ok; ++it) {
        const int64_t m0 = ((int64_t)cl + (int64_t)it * ncl) * kBN;
        const int64_t rem = a.M - m0 - col_lo;
        const int valid = rem <= 0 ? 0 : (rem >= kRows ? kRows : (int)rem);
        if (YS) {
          ok = wait_bar(ptx::smem_addr(&y_full[it & 1]), (it >> 1) & 1, abort_flag, a.status);
          ok = __all_sync(0xffffffffu, ok);   // the warp arrives as one
          if (!ok) break;
        }
        const float* yt = YS ? ys + (it & 1) * kBN + col_lo : a.y + m0 + col_lo;
        for (int c = 0; c < Cp; ++c) {
          const uint32_t buf = acc_it & 1, u = acc_it >> 1;
          const int chrom = c * 2 * kRows + (int)rank * kRows + row;
          const float bias = bias_n;
          bias_n = a.a0[(c + 1 == Cp ? 0 : c + 1) * 2 * kRows + (int)rank * kRows + row];
          last.begin();
          float4 ya[4];
          if (valid >= 32) epi_targets<YS>(yt, ya);
          ok = wait_bar(ptx::smem_addr(&acc_full[buf]), u & 1, abort_flag, a.status);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          ptx::tc_fence_after();
          float2 sum;
          float tail;
          epi_reduce<false, ABS, YS>(tmem + lane_addr + buf * (uint32_t)kBN + (uint32_t)col_lo, yt,
                                     valid, ya, bias, -1.f, last, sum, tail);
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(acc_empty_lead0 + 8 * buf);
          last.sum = sum;
          last.tail = tail;
          last.row = part_row + chrom;
          last.first = it == 0;
          ++acc_it;
        }
        if (YS && ok) {
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(ptx::smem_addr(&y_empty[it & 1]));
        }
      }
      if (ok) {
        last.begin();
        last.end();
      }
    };
    if (a.ycopy) reduce_tiles(std::true_type{});
    else reduce_tiles(std::false_type{});
  } else {
    // ---------------- expansion (both CTAs) ----------------
    const int bt = threadIdx.x - kBasisWarp0 * 32;
    const int r0 = bt & (kRows - 1), grp = bt >> 7;   // this thread's pattern row, warpgroup
    for (int cid = bt; cid < KB * 8; cid += kBasisThreads)
      tab[cid] = chunk_desc(cid, a.basis, a.d, a.Kp);
    ptx::named_bar(1, kBasisThreads);
    const uint32_t phi_full_lead0 = ptx::mapa(ptx::smem_addr(phi_full), 0);
    // (whole features at a time: see expand_stream.cuh)
    const bool stream = a.xstage && stream_degree(a.d);
    if (stream) {
      StreamArgs sa;
      sa.phi = ptx::smem_addr(phi);
      sa.slot_bytes = kRows * 128;
      sa.lo_off = 0;
      sa.phi_full0 = phi_full_lead0;
      sa.phi_free0 = ptx::smem_addr(phi_free);
      sa.x_full = ptx::smem_addr(x_full);
      sa.x_empty = ptx::smem_addr(x_empty);
      sa.xs = xs;
      sa.cs = nullptr;
      sa.xstride = kRows;
      sa.xblocks = 0;   // one block of 128 rows
      sa.N = N;
      sa.KB = KB;
      sa.NS = NS;
      sa.RW = kRows / 2;
      sa.R = 2;
      sa.QS = 2 * kBasisThreads / kRows;
      sa.bt = bt;
      sa.my_tiles = my_tiles;
      sa.abort_flag = abort_flag;
      sa.status = a.status;
      stream_dispatch<kFormBF16, true>(a.basis, a.d, sa);
    }
    auto slot_free = [&](int q) -> bool {
      const int use = q / NS;
      return use == 0 ||
             wait_bar(ptx::smem_addr(&phi_free[q % NS]), (use - 1) & 1, abort_flag, a.status);
    };
    auto publish = [&](int q) {
      ptx::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive_cluster(phi_full_lead0 + 8 * (q % NS));
    };
    bool ok = true;
    if (!a.xstage) {
      // Chebyshev runs of 8 degrees, features read from global memory (L2):
      // the x of a K-block's 8 chunks are loaded one K-block ahead; thread 0
      // prefetches this CTA's feature block of the tile after next into L2
      auto xptr = [&](int itn) -> const float* {
        const int64_t blk = ((int64_t)cl + (int64_t)itn * ncl) * 2 + rank;
        return a.Xt + blk * (int64_t)N * kPatBlock + r0;
      };
      auto prefetch_tile = [&](int itn) {
        const int64_t blk = ((int64_t)cl + (int64_t)itn * ncl) * 2 + rank;
        ptx::bulk_prefetch_l2(a.Xt + blk * N * kPatBlock, (uint32_t)(N * kPatBlock * 4));
      };
      // The two warpgroups take the K-blocks in turn. (Not with one slot: a
      // group would await the second release ahead, which a parity cannot tell.)
      const int ngr = NS > 1 ? 2 : 1;
      const int nq = grp < ngr ? my_tiles * KB : 0;
      float nx[8];
      auto load_kb = [&](int itn, int kbn) {
        const float* p = xptr(itn);
#pragma unroll
        for (int q = 0; q < 8; ++q) nx[q] = __ldg(p + chunk_feature(tab[kbn * 8 + q]) * kPatBlock);
      };
      if (bt == 0) {
        if (my_tiles > 0) prefetch_tile(0);
        if (my_tiles > 1) prefetch_tile(1);
      }
      if (grp < nq) load_kb(grp / KB, grp % KB);
      int fetched = 0;   // tiles whose successor but one is prefetched
      for (int q = grp; q < nq; q += ngr) {
        const int it = q / KB, kb = q - it * KB;
        if (bt == 0)
          for (; fetched <= it; ++fetched)
            if (fetched + 2 < my_tiles) prefetch_tile(fetched + 2);
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = nx[e];
        if (q + ngr < nq) load_kb((q + ngr) / KB, (q + ngr) % KB);
        ok = slot_free(q);
        if (!ok) break;
        uint8_t* phik = phi + (size_t)(q % NS) * kRows * 128;
#pragma unroll
        for (int qd = 0; qd < 8; qd += 2) {
          const uint32_t da = tab[kb * 8 + qd], db = tab[kb * 8 + qd + 1];
          float va[8], vb[8];
          cheb_run_pair(x[qd], chunk_degree(da), x[qd + 1], chunk_degree(db),
                        va, vb);
          if (da & kChunkZero) {
#pragma unroll
            for (int e = 0; e < 8; ++e) va[e] = 0.f;
          }
          if (db & kChunkZero) {
#pragma unroll
            for (int e = 0; e < 8; ++e) vb[e] = 0.f;
          }
          store_bf16x8(phik, r0, qd, va);
          store_bf16x8(phik, r0, qd + 1, vb);
        }
        publish(q);
      }
    } else if (!stream) {
      const float* xrow = xs + r0;   // block layout [N][128]
      for (int it = 0; it < my_tiles && ok; ++it) {
        ok = wait_bar(ptx::smem_addr(x_full), it & 1, abort_flag, a.status);
        if (!ok) break;
        for (int kb = 0; kb < KB; ++kb) {
          const int q = it * KB + kb;
          ok = slot_free(q);
          if (!ok) break;
          uint8_t* phik = phi + (size_t)(q % NS) * kRows * 128;
#pragma unroll 1
          for (int qd = 4 * grp; qd < 4 * grp + 4; qd += 2) {
            float va[8], vb[8];
            gen8(tab[kb * 8 + qd], a.basis, a.d, N, xrow, kRows, va);
            gen8(tab[kb * 8 + qd + 1], a.basis, a.d, N, xrow, kRows, vb);
            store_bf16x8(phik, r0, qd, va);
            store_bf16x8(phik, r0, qd + 1, vb);
          }
          publish(q);
        }
        if (!ok) break;
        ptx::mbar_arrive(ptx::smem_addr(x_empty));
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();   // the pair's MMAs, loads and remote arrivals are over
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc2(tmem, 512u);
  }
}

}  // namespace

TcPlan plan_tc_pair(const Shape& s, int P, int num_sms) {
  TcPlan pl{};
  pl.form = kFormBF16;
  pl.pair = 1;
  pl.KB = ceil_div(s.Kp, 64);
  pl.C = 2 * ceil_div(P, kBN);
  pl.BN = kBN;
  pl.ok = false;
  if (num_sms < 2) return pl;
  // features from L2 for Chebyshev runs of 8 degrees (the x of a chunk is one
  // load), else staged
  const int xstage = (s.basis == GAME_BASIS_CHEB && s.d % 8 == 0) ? 0 : 1;
  for (int stages = 4; stages >= 3 && !pl.ok; --stages)
    for (int NS = 2 * pl.KB; NS >= pl.KB && !pl.ok; --NS) {
      const int sm = smem_plan2(pl.KB, NS, s.N, stages, xstage, 0).total;
      if (sm <= kMaxSmem) {
        pl.NS = NS;
        pl.stages = stages;
        pl.xstage = xstage;
        pl.smem_bytes = sm < kMinSmem ? kMinSmem : sm;
        pl.ok = true;
      }
    }
  if (!pl.ok) return pl;
  {
    const int sm = smem_plan2(pl.KB, pl.NS, s.N, pl.stages, xstage, 1).total;
    if (sm <= kMaxSmem) {
      pl.ycopy = 1;
      if (pl.smem_bytes < sm) pl.smem_bytes = sm;
    }
  }
  const int ntiles = ceil_div(s.M, kBN);
  const int clusters = ntiles < num_sms / 2 ? ntiles : num_sms / 2;
  pl.grid = 2 * clusters;
  pl.tmem_cols = 512;
  pl.rows = 2 * clusters;   // one partial row per (cluster, column half)
  return pl;
}

cudaError_t launch_fitness_tc_pair(const TcPlan& pl, const Shape& s, const float* Xt,
                                   const float* y, const uint8_t* popA, const float* a0, int Ppad,
                                   double* part, int* status, int err, cudaStream_t st) {
  if (!pl.ok || !pl.pair || pl.form != kFormBF16) return cudaErrorInvalidValue;
  if (pl.NS < pl.KB || pl.NS > 2 * pl.KB || pl.grid % 2 != 0 || Ppad < pl.C * 128)
    return cudaErrorInvalidValue;
  Tc2Args a;
  a.M = s.M;
  a.N = s.N;
  a.d = s.d;
  a.basis = s.basis;
  a.Kp = s.Kp;
  a.KB = pl.KB;
  a.Cp = pl.C / 2;
  a.NS = pl.NS;
  a.stages = pl.stages;
  a.xstage = pl.xstage;
  a.ycopy = pl.ycopy;
  const int last_cols = s.Kp - 64 * (pl.KB - 1);
  a.nmma_last = (last_cols + 15) / 16;
  a.ntiles = ceil_div(s.M, kBN);
  a.Ppad = Ppad;
  a.Xt = Xt;
  a.y = y;
  a.popA = popA;
  a.a0 = a0;
  a.part = part;
  a.status = status;
  a.stall_ns = hook_take_stall_ns();
  void (*kern)(const Tc2Args) =
      err == GAME_ERR_MAE ? fitness_tc2_kernel<true> : fitness_tc2_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       pl.smem_bytes);
  if (e != cudaSuccess) return e;
  return launch_behind(kern, pl.grid, kThreads, pl.smem_bytes, st, a);
}

}  // namespace game
