// expand_stream.cuh -- the expansion role of the tensor-core fitness kernels
// with the basis and the degree compile-time constants (degrees 1..10).
//
// What bounds it: eight warps, two per scheduler, produce every expansion value
// of the SM, so the instructions per value decide. The chunk generator it
// replaces for these degrees decoded a descriptor per 8 columns, restarted the
// feature's recurrence there (for the trigonometric basis with another sincosf
// per chunk) and tested the end of a run at every value: at M = 10^6, N = 32,
// trigonometric degree 8, P = 1024 (SM pairs) the BF16 evaluation took 2.58 ms, 0.84
// with this file on four warps, 0.56 on eight (1.88 PFLOP/s). Here a thread takes
// whole features: the shortest run
// of them that fills whole 16-byte units (8 columns, 16 in FP8) is one group,
// its values are straight-line code (one start per feature, one FMA per
// value), rounded and packed in registers, then stored unit by unit.
// Values are those of gen_chunk bit for bit: the same operations from the same
// start values.
//
// Work split: a thread owns R rows of the tile (row passes RW apart) and every
// QS-th group, so the threads of a row move through the K-blocks together and
// a K-block is complete after about G QS columns' time. Before its first store
// into a K-block a thread awaits the release of the K-block's slot by the MMAs
// that read its previous use; it arrives on a K-block once it has no group left
// in it.
#pragma once
#include "basis.cuh"
#include "game_internal.cuh"
#include "tc_common.cuh"
#include "tc_ptx.cuh"

namespace game {
namespace tc {

struct StreamArgs {
  uint32_t phi;         // shared address of expansion slot 0
  uint32_t slot_bytes;  // one K-block slot (hi and lo images for bf16x3)
  uint32_t lo_off;      // bf16x3: lo image inside a slot
  uint32_t phi_full0;   // arrivals (pairs: the even CTA's barriers, cluster address)
  uint32_t phi_free0;
  uint32_t x_full, x_empty;
  const float* xs;      // staged features: row r, feature i at xs[xoff(r) + i xstride]
  const float* cs;      // FP8 column scales
  int xstride, xblocks; // xblocks: rows in 128-row blocks of N features
  int N, KB, NS;
  int RW, R, QS;        // rows per pass, passes, threads per row
  int bt;               // thread of the role, 0..255
  int my_tiles;
  volatile int* abort_flag;
  int* status;
};

// K-block sequence number q (over all tiles) with its slot and the slot's use count
struct SlotWalk {
  int q, slot, use;
  __device__ __forceinline__ void next(int NS) {
    ++q;
    if (++slot == NS) {
      slot = 0;
      ++use;
    }
  }
};

template <int F, int BASIS, int D>
struct StreamGroup {
  static constexpr int W = (BASIS == GAME_BASIS_TRIG ? 2 : 1) * D;   // columns per feature
  static constexpr int UC = form_cols(F) / 8;                        // columns per 16-byte unit
  // features per group: whole units, and at least three of them where that
  // takes no more than 8 features (the K-block bookkeeping is per group)
  static constexpr int NF0 = UC / const_gcd(W, UC), CH0 = NF0 * W / UC;
  static constexpr int MU = CH0 >= 3 || NF0 > 4 ? 1 : (CH0 == 2 || NF0 == 4 ? 2 : 4);
  static constexpr int NF = NF0 * MU;
  static constexpr int CH = NF * W / UC;                             // units per group
  static constexpr int NW = 4 * CH * form_nphi(F);                   // packed words per row
  // two rows at a time where a group alone has few independent recurrences
  static constexpr int RU = (NF < 4 && 2 * NW <= 48) ? 2 : 1;
};

// One row's group: the values of features x[0..NF), packed. w[4 u ..] unit u
// (bf16x3: the lo image's words after all of the hi image's). TAIL: only the
// first nf features are there, the others' columns are zero; without it the
// features are straight-line code whose recurrences interleave (trigonometric
// features are separate blocks anyway, sincosf branches on large arguments).
template <int F, int BASIS, int D, bool TAIL>
__device__ __forceinline__ void stream_values(
    const float (&x)[StreamGroup<F, BASIS, D>::NF], const float* cs, int u0, int units, int nf,
    uint32_t (&w)[StreamGroup<F, BASIS, D>::NW]) {
  using SG = StreamGroup<F, BASIS, D>;
  float v[4];             // columns of the word being packed
  float4 sc[4] = {};      // FP8: the scales of the unit's columns
#pragma unroll
  for (int f = 0; f < SG::NF; ++f) {
    float val[SG::W];
    if (TAIL && f >= nf) {
#pragma unroll
      for (int e = 0; e < SG::W; ++e) val[e] = 0.f;
    } else {
      float fm = 1.f, fv = x[f], c2, s1 = 0.f;   // f_{j-1}, f_j
      if (BASIS == GAME_BASIS_TRIG) {
        float c1;
        sincosf(x[f], &s1, &c1);
        fv = c1;
      }
      c2 = fv + fv;
#pragma unroll
      for (int e = 0; e < SG::W; ++e) {
        if (e > 0) {
          if (BASIS == GAME_BASIS_TRIG && e == D) {
            fm = 0.f;   // sin(0 x)
            fv = s1;
          } else {
            const float fn = fmaf(c2, fv, -fm);
            fm = fv;
            fv = fn;
          }
        }
        val[e] = fv;
      }
    }
#pragma unroll
    for (int e = 0; e < SG::W; ++e) {
      const int c = f * SG::W + e;
      if (F == kFormFP8) {
        if ((c & 15) == 0) {
          // (units past the last K-block are dropped: their scales are not read)
          const int u = u0 + (c >> 4);
          const float4* s4 = reinterpret_cast<const float4*>(cs) + (u < units ? u * 4 : 0);
#pragma unroll
          for (int h = 0; h < 4; ++h) sc[h] = s4[h];
        }
        const float4 s4 = sc[(c >> 2) & 3];
        v[c & 3] = val[e] * ((c & 3) == 0 ? s4.x : (c & 3) == 1 ? s4.y : (c & 3) == 2 ? s4.z : s4.w);
        if ((c & 3) == 3) w[c >> 2] = e4m3x4_bits(v[0], v[1], v[2], v[3]);
      } else {
        v[c & 1] = val[e];
        if (c & 1) {
          if (F == kFormBF16) w[c >> 1] = bf16x2_bits(v[0], v[1]);
          else split_bf16x2(v[0], v[1], w[c >> 1], w[4 * SG::CH + (c >> 1)]);
        }
      }
    }
  }
}

// The whole expansion role of one thread. PAIR: arrivals go to the even CTA's
// barriers, one per warp.
template <int F, int BASIS, int D, bool PAIR>
__device__ __noinline__ void stream_expand(const StreamArgs a) {
  using SG = StreamGroup<F, BASIS, D>;
  constexpr int NPHI = form_nphi(F);
  const int N = a.N, KB = a.KB, NS = a.NS, R = a.R, QS = a.QS;
  const int r0 = a.bt % a.RW, q0 = a.bt / a.RW;
  const int ng = (N + SG::NF - 1) / SG::NF;
  const int units = KB * 8;
  SlotWalk fr{0, 0, 0}, ar{0, 0, 0};   // next K-block to await, to arrive on
  bool ok = true;
  auto await = [&](int q) {   // the slots of K-blocks up to q are free
    if (fr.q > q) return;
    while (ok && fr.q <= q) {
      if (fr.use > 0)
        ok = wait_bar(a.phi_free0 + 8u * (uint32_t)fr.slot, (uint32_t)(fr.use - 1) & 1u,
                      a.abort_flag, a.status);
      fr.next(NS);
    }
    if (PAIR) ok = __all_sync(0xffffffffu, ok);   // the warp arrives as one
  };
  auto arrive_below = [&](int qend) {
    if (ar.q >= qend) return;
    ptx::fence_proxy_async_smem();
    if (PAIR) __syncwarp();
    while (ok && ar.q < qend) {
      await(ar.q);
      if (!ok) return;
      if (!PAIR) ptx::mbar_arrive(a.phi_full0 + 8u * (uint32_t)ar.slot);
      else if ((threadIdx.x & 31) == 0)
        ptx::mbar_arrive_cluster(a.phi_full0 + 8u * (uint32_t)ar.slot);
      ar.next(NS);
    }
  };
  auto xrow = [&](int r) -> const float* {
    return a.xblocks ? a.xs + (r >> 7) * N * 128 + (r & 127) : a.xs + r;
  };
  auto load_x = [&](const float* xr, int g, float (&x)[SG::NF]) {
#pragma unroll
    for (int f = 0; f < SG::NF; ++f) {
      const int i = g * SG::NF + f;
      x[f] = i < N ? xr[i * a.xstride] : 0.f;
    }
  };
  for (int it = 0; it < a.my_tiles; ++it) {
    ok = wait_bar(a.x_full, it & 1, a.abort_flag, a.status);
    if (PAIR) ok = __all_sync(0xffffffffu, ok);
    if (!ok) return;
    const int qbase = it * KB;
    SlotWalk gs = ar;   // K-block of the group's first unit (ar.q == qbase here)
    for (int g = q0; g < ng; g += QS) {
      const int u0 = g * SG::CH;
      while (gs.q < qbase + (u0 >> 3)) gs.next(NS);
      const int nf = N - g * SG::NF;   // features from the group's first on
#pragma unroll 1
      for (int rr = 0; rr < R; rr += SG::RU) {
        uint32_t w[SG::RU][SG::NW];
        uint32_t row[SG::RU], sw[SG::RU];
#pragma unroll
        for (int b = 0; b < SG::RU; ++b) {
          // (an odd last row is taken twice: the same values to the same place)
          const int r = r0 + (rr + b < R ? rr + b : rr) * a.RW;
          float x[SG::NF];
          load_x(xrow(r), g, x);
          if (BASIS == GAME_BASIS_TRIG || (SG::NF > 1 && nf < SG::NF))
            stream_values<F, BASIS, D, true>(x, a.cs, u0, units, nf, w[b]);
          else
            stream_values<F, BASIS, D, false>(x, a.cs, u0, units, nf, w[b]);
          row[b] = (uint32_t)r * 128u;
          sw[b] = (uint32_t)(r & 7) << 4;
        }
        SlotWalk sk = gs;
        await(sk.q);
        if (!ok) return;
        uint32_t kaddr = a.phi + (uint32_t)sk.slot * a.slot_bytes;
        bool live = true;
#pragma unroll
        for (int q = 0; q < SG::CH; ++q) {
          const int u = u0 + q;
          if (q > 0 && (u & 7) == 0) {   // the next K-block
            live = u < units;
            if (live) {
              sk.next(NS);
              await(sk.q);
              if (!ok) return;
              kaddr = a.phi + (uint32_t)sk.slot * a.slot_bytes;
            }
          }
          if (!live) continue;
          const uint32_t pos = (uint32_t)(u & 7) << 4;
#pragma unroll
          for (int b = 0; b < SG::RU; ++b)
#pragma unroll
            for (int im = 0; im < NPHI; ++im) {
              const int k = 4 * (im * SG::CH + q);
              ptx::st_shared_v4(kaddr + (im ? a.lo_off : 0u) + row[b] + (pos ^ sw[b]),
                                make_uint4(w[b][k], w[b][k + 1], w[b][k + 2], w[b][k + 3]));
            }
        }
      }
      const int next_kb = ((g + QS) * SG::CH) >> 3;
      arrive_below(qbase + (next_kb < KB ? next_kb : KB));
      if (!ok) return;
    }
    // zero units from the end of the last group to the end of the last K-block
    if (q0 == ng % QS) {
      for (int u = ng * SG::CH; u < units; ++u) {
        while (gs.q < qbase + (u >> 3)) gs.next(NS);
        await(gs.q);
        if (!ok) return;
        for (int rr = 0; rr < R; ++rr) {
          const int r = r0 + rr * a.RW;
#pragma unroll
          for (int im = 0; im < NPHI; ++im)
            ptx::st_shared_v4(a.phi + (uint32_t)gs.slot * a.slot_bytes + (im ? a.lo_off : 0u) +
                                  (uint32_t)r * 128u +
                                  ((uint32_t)((u & 7) ^ (r & 7)) << 4),
                              make_uint4(0u, 0u, 0u, 0u));
        }
      }
    }
    arrive_below(qbase + KB);
    if (!ok) return;
    ptx::mbar_arrive(a.x_empty);
  }
}

// true when stream_expand covers the degree (the caller's generic generator
// serves the others)
__host__ __device__ constexpr bool stream_degree(int d) { return d >= 1 && d <= 10; }

template <int F, bool PAIR>
__device__ __forceinline__ void stream_dispatch(int basis, int d, const StreamArgs& a) {
#define GAME_STREAM_CASE(D)                                                      \
  case D:                                                                        \
    if (basis == GAME_BASIS_CHEB) stream_expand<F, GAME_BASIS_CHEB, D, PAIR>(a); \
    else stream_expand<F, GAME_BASIS_TRIG, D, PAIR>(a);                          \
    break;
  switch (d) {
    GAME_STREAM_CASE(1)
    GAME_STREAM_CASE(2)
    GAME_STREAM_CASE(3)
    GAME_STREAM_CASE(4)
    GAME_STREAM_CASE(5)
    GAME_STREAM_CASE(6)
    GAME_STREAM_CASE(7)
    GAME_STREAM_CASE(8)
    GAME_STREAM_CASE(9)
    GAME_STREAM_CASE(10)
  }
#undef GAME_STREAM_CASE
}

}  // namespace tc
}  // namespace game
