// Factor chain of Algorithm 2, Phase 3 on pairs of SMs (tcgen05 cta_group::2), for the kind::f16
// forms (FP16, BF16 and their split forms) with d >= 2.
//
// A cluster of two CTAs takes 256 consecutive points of one side, 128 per CTA. Chain step 1
// (n -> R_1, a few hundred FMAs per point) runs on the FP32 pipe; every later step
//   S_out (256 x R_out) = A (256 x K) * Gs (K x R_out),  A[p, j + np a] = S_in[p, a] T_j(xhat_p)
// is one M = 256 MMA chain: A generated by sixteen warps per CTA straight into tensor memory
// (128 lanes = that CTA's points), half of the core's columns in each CTA's shared memory, the
// accumulator in tensor memory.
//
// Why this shape. The shared-memory form (chain_tce_kernel) moves, per 64 values of K at N = 192,
// 32 KB of generated A in, 32 KB of S out, 48 KB of core in, and 120 KB of MMA operand reads:
// about 1,860 of its 2,300 clocks per chunk at 128 B/clock, against 1,150 clocks of MMA. With A in
// tensor memory and the core split over two SMs, shared memory carries 24 KB of core in and 36 KB
// of operand reads, and L2 delivers half as many core bytes per point, so the tensor pipe is what is
// left. K runs over a slowest (chunks of 4 values of a, np = n rounded up to a multiple of 4):
// n = 12, 16, 20 then need no padding in j, and a generator thread holds its point's T_j in
// registers and reads one S_in value per a.
//
// The order of work hides the hand-offs: with two tensor-core steps (d = 3) the first one of item
// t + 1 is issued before the last one of item t, so reading S back, and the output of item t - 1
// leaving its accumulator, run behind MMAs. K goes through in quads of four values of a. The four
// generator warps of a lane quarter take every fourth quad each, counted through all steps: a
// warp then has four quads' time for the waits, fences and arrivals of one, and S_in stays private to
// the thread that wrote it. (With every warp at work on every quad, the serial part of one
// quad, about 900 clocks, set the pace: 6.9 ms on 1024 d = 2 instances.)
//
// Measured (3xFP16, against the shared-memory kernel): ranks 9, 44, 177 | 180, 49, 10, n = 12, a
// million points a side 1.673 -> 0.819 ms (its MMAs alone take 0.56 ms), 1024 instances with ranks 10, 63 |
// 63, 12, n = 20, 22M points a side 19.2 -> 4.30 ms (generation bound: 3.5 ms without the conversions).
//
// Warps per CTA: 0 streams the core's quads by cp.async.bulk; 1 issues the MMAs (CTA 0) or passes on
// the arrival of CTA 1's quads; 3 streams the points; 4..19 generate; 20..23 write the output, through
// shared memory and one bulk copy per 32 rows. Quads of A (tensor memory), quads of the core and
// tiles of points (shared memory) have rings of their own.
// Barriers: full_a[s] in CTA 0 (the quad's 4 warps in each CTA), full_b[s] in CTA 0 (both CTAs' core
// quads) and in CTA 1 (its own); empty_a[s], empty_b[s], mid, last_done[r] committed to both CTAs;
// d2free, rfree[r] in CTA 0 (every reader warp of both CTAs); xfull[s], xempty[s] within a CTA. Once
// a wait has run out its role goes on without waiting: what it writes is its own CTA's memory.
// Waits are bounded as in chain_tc.cu: on running out, PTTK_ETIMEOUT in the status word, no new
// MMAs or copies, and the CTAs still meet at the end.
#include <stdio.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "chain_pair.cuh"
#include "tcgen05.cuh"

namespace pttk {
namespace {

constexpr int PAIR_GEN = 16, PAIR_EPI = 4;
constexpr int PAIR_THREADS = 32 * (4 + PAIR_GEN + PAIR_EPI);
constexpr int PAIR_MAX_NS = 8;               // deepest ring
constexpr int PAIR_XD = 4;                   // tiles of points in flight

struct PairStep {
  const uint8_t* img;      // nquads x 2 CTAs x parts x (Npad / 2 rows x 4 np values)
  uint32_t bytes, idesc;   // bytes of one quad of one CTA
  int nquads, R_out, Npad, coord;  // nquads: quads of four values of a
  float lo, hi;
  float in_scale;          // power of two on S_in as stored for this step
  float out_scale;         // power of two that unscales the accumulator
};
struct PairArgs {
  PairStep st[2][2];
  int ntc, n, np, d;
  const float* g1[2];      // first core, n x r1 column-major, FP32
  int r1[2], c1[2];
  float lo1[2], hi1[2];
  int64_t N[2], P0, npairs;
  const float* pts[2];
  float* out[2];
  int* status;
  int r1_pad, s2_rows;     // rows of the S_1 and S_2 buffers (multiples of 16)
  int stage_cols;          // widest output row
  int nd, d_cols, d2_col, a_col, slot_cols, na, nb;  // na A slots, nb core slots
  uint32_t b_slot;
};

__device__ __forceinline__ void pair_umma(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void pair_commit(uint64_t* bar) {  // arrives in both CTAs
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
// Arrive on CTA 0's barrier at this offset. The default (CTA-scope) release: what the arrival hands
// over is tensor memory, ordered by the tcgen05 fences around it, or a core chunk, ordered by the copy's
// own barrier. A cluster-scope release would wait for every outstanding store of the warp (over 1,000
// clocks per arrival: d = 3 chain 1.43 -> 1.33 ms without it).
__device__ __forceinline__ void arrive_cta0(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, 0;\n\t"
      "mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}\n" ::"r"(smem_u32(bar))
      : "memory");
}

// Position in a ring: slot and the parity of its current round.
struct Ring {
  uint32_t slot = 0, par = 0;
  __device__ __forceinline__ void next(uint32_t n) {
    if (++slot == n) {
      slot = 0;
      par ^= 1;
    }
  }
  __device__ __forceinline__ void skip(uint32_t m, uint32_t n) {
    slot += m;
    while (slot >= n) {
      slot -= n;
      par ^= 1;
    }
  }
};

template <int W>
__device__ __forceinline__ void tmem_st(uint32_t c, const uint32_t* v) {
  if constexpr (W == 2)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(c), "r"(v[0]), "r"(v[1]) : "memory");
  else if constexpr (W == 4)
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(c), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3])
                 : "memory");
  else
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(c), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
// COLS (even) consecutive columns in as few stores as there are powers of two in COLS
template <int COLS>
__device__ __forceinline__ void tmem_st_cols(uint32_t c, const uint32_t* v) {
  if constexpr (COLS >= 8) {
    tmem_st<8>(c, v);
    tmem_st_cols<COLS - 8>(c + 8, v + 8);
  } else if constexpr (COLS >= 4) {
    tmem_st<4>(c, v);
    tmem_st_cols<COLS - 4>(c + 4, v + 4);
  } else if constexpr (COLS >= 2) {
    tmem_st<2>(c, v);
  }
}
// four consecutive columns of this warp's lanes, and the wait for them
__device__ __forceinline__ float4 tmem_ld4(uint32_t c) {
  uint32_t r[4];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
      : "r"(c)
      : "memory");
  return make_float4(__uint_as_float(r[0]), __uint_as_float(r[1]), __uint_as_float(r[2]), __uint_as_float(r[3]));
}

// Packed FP32 pairs (the Blackwell two-wide FP32 instructions).
__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t x, uint64_t y) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t x, uint64_t y, uint64_t z) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  return r;
}

// T_0 .. T_{NP-1} at x on [lo, hi] (zero from n on), as pairs in registers.
template <int NP>
__device__ __forceinline__ void cheb_regs(float x, float lo, float hi, int n, uint64_t* T2) {
  const float xh = (2.f * x - lo - hi) / (lo - hi);
  const float x2 = 2.f * xh;
  float T[NP];
  T[0] = 1.f;
  T[1] = xh;
#pragma unroll
  for (int k = 2; k < NP; ++k) T[k] = x2 * T[k - 1] - T[k - 2];
#pragma unroll
  for (int k = NP - 3; k < NP; ++k)
    if (k >= n) T[k] = 0.f;
#pragma unroll
  for (int k = 0; k < NP / 2; ++k) T2[k] = pack2(T[2 * k], T[2 * k + 1]);
}

// The NP values v = S T_j of one a into tensor memory: h = fl16(v) as 16-bit pairs from column `hi`, and
// for the split forms fl16(h - v) from column `lo` (its MMA negates A). The residual is taken from
// the exact product by one fused multiply-add.
template <int FMT, bool SPLIT, int NP>
__device__ __forceinline__ void gen_a(float s, const uint64_t* T2, uint32_t hi, uint32_t lo) {
  const uint64_t s2 = pack2(s, s), m2 = pack2(-s, -s);
  uint32_t h[NP / 2], l[NP / 2];
#pragma unroll
  for (int q = 0; q < NP / 2; ++q) {
    const float2 v = unpack2(mul2(s2, T2[q]));
    float2 hf;
    if constexpr (FMT == FMT_BF16) {
      const __nv_bfloat162 hb = __floats2bfloat162_rn(v.x, v.y);
      h[q] = *reinterpret_cast<const uint32_t*>(&hb);
      hf = __bfloat1622float2(hb);
    } else {
      const __half2 hb = __floats2half2_rn(v.x, v.y);
      h[q] = *reinterpret_cast<const uint32_t*>(&hb);
      hf = __half22float2(hb);
    }
    if constexpr (SPLIT) {
      const float2 r = unpack2(fma2(m2, T2[q], pack2(hf.x, hf.y)));
      if constexpr (FMT == FMT_BF16) {
        const __nv_bfloat162 lb = __floats2bfloat162_rn(r.x, r.y);
        l[q] = *reinterpret_cast<const uint32_t*>(&lb);
      } else {
        const __half2 lb = __floats2half2_rn(r.x, r.y);
        l[q] = *reinterpret_cast<const uint32_t*>(&lb);
      }
    }
  }
  tmem_st_cols<NP / 2>(hi, h);
  if (SPLIT) tmem_st_cols<NP / 2>(lo, l);
}

// Shared-memory pointers and the launch's constants, as every warp role needs them.
struct PairCtx {
  uint8_t* b_base;
  float *S1, *S2, *G1, *stage, *X;
  const PairStep* steps;
  uint64_t *full_a, *full_b, *empty_a, *empty_b, *xfull, *xempty, *mid, *d2free, *last_done, *rfree;
  volatile int* abort_flag;
  uint32_t tmem, rank;
  int64_t it0, itstep;
  __device__ __forceinline__ int side(const PairArgs& a, int64_t it) const { return it < a.P0 ? 0 : 1; }
  __device__ __forceinline__ int64_t row0(const PairArgs& a, int64_t it) const {
    return (it - (it < a.P0 ? 0 : a.P0)) * (2 * TILE_M) + (int64_t)rank * TILE_M;
  }
};

// One generator thread: point row `row` of its CTA, the quads whose running number is `part` mod 4.
template <int FMT, bool SPLIT, int NP>
__device__ __forceinline__ void pair_generate(const PairArgs& a, const PairCtx& c) {
  constexpr uint32_t LO = 2 * NP;  // tensor-memory columns from a quad's high parts to its residuals
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quarter = warp & 3, part = (warp - 4) >> 2;
  const int row = 32 * quarter + lane;
  const uint32_t lanes = (uint32_t)(32 * quarter) << 16;
  const int ntc = a.ntc, n = a.n, d = a.d;
  const uint32_t na = (uint32_t)a.na;
  // this thread's own S values, its k-th quad's four at [(4 k + i) TILE_M]: which warp takes a quad
  // changes from item to item, so the buffers are split by warp and not by quad
  float* s1 = c.S1 + (size_t)part * (a.r1_pad / 4) * TILE_M + row;
  float* s2 = c.S2 + (size_t)part * (a.s2_rows / 4) * TILE_M + row;
  const uint32_t col0 = c.tmem + lanes + (uint32_t)a.a_col;
  const float* xrow = c.X + row * d;
  Ring ra, rx;             // slot of quad number g; slot of the newest tile of points read
  int g = 0;               // running number of the next step's first quad, mod 4
  uint32_t midpar = 0;
  bool dead = false;
  uint64_t T2[NP / 2];
  auto wait = [&](uint64_t* bar, uint32_t par) {
    if (!dead) dead = !mbar_wait(bar, par, c.abort_flag);
    __syncwarp();
  };
  auto first_quad = [&](int base) { return (part - base) & 3; };
  // S_1 = B_1 G_1 for the values of this warp's quads, scaled
  auto first_step = [&](int sd, float x) {
    const int nq = c.steps[sd * 2].nquads;
    int q = first_quad(g);
    if (q >= nq) return;
    cheb_regs<NP>(x, a.lo1[sd], a.hi1[sd], n, T2);
    const float sc = c.steps[sd * 2].in_scale;
    for (float* s = s1; q < nq; q += 4, s += 4 * TILE_M) {
      const float* G = c.G1 + (size_t)(sd * a.r1_pad + 4 * q) * NP;
#pragma unroll
      for (int i = 0; i < 4; ++i, G += NP) {
        uint64_t u = pack2(0.f, 0.f), v = u;
#pragma unroll
        for (int k = 0; k < NP / 4; ++k) {
          const ulonglong2 w = reinterpret_cast<const ulonglong2*>(G)[k];
          u = fma2(T2[2 * k], w.x, u);
          v = fma2(T2[2 * k + 1], w.y, v);
        }
        const float2 x0 = unpack2(u), x1 = unpack2(v);
        s[i * TILE_M] = ((x0.x + x0.y) + (x1.x + x1.y)) * sc;
      }
    }
  };
  auto generate = [&](int sd, int si, const float* s, float x) {
    const PairStep& st = c.steps[sd * 2 + si];
    const int nq = st.nquads;
    int q = first_quad(g);
    if (q < nq) {
      cheb_regs<NP>(x, st.lo, st.hi, n, T2);
      Ring r = ra;
      r.skip((uint32_t)q, na);
      for (; q < nq; q += 4, s += 4 * TILE_M) {
        float v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = s[i * TILE_M];
        wait(&c.empty_a[r.slot], r.par ^ 1);
        tc_fence_after();
        const uint32_t col = col0 + r.slot * (uint32_t)a.slot_cols;
#pragma unroll
        for (int i = 0; i < 4; ++i) gen_a<FMT, SPLIT, NP>(v[i], T2, col + i * (NP / 2), col + LO + i * (NP / 2));
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_cta0(&c.full_a[r.slot]);
        r.skip(4, na);
      }
    }
    ra.skip((uint32_t)nq, na);
    g = (g + nq) & 3;
  };
  // the points of the next item in this warp's order
  auto next_points = [&](bool first) -> const float* {
    if (!first) rx.next(PAIR_XD);
    wait(&c.xfull[rx.slot], rx.par);
    return xrow + rx.slot * (uint32_t)(TILE_M * d);
  };
  const float *xc = xrow, *xn = xrow;  // points of the item at hand, and of the next one
  if (c.it0 < a.npairs) {
    xc = next_points(true);
    if (ntc == 2) {
      const int sd = c.side(a, c.it0);
      first_step(sd, xc[a.c1[sd]]);
      generate(sd, 0, s1, xc[c.steps[sd * 2].coord]);
    }
  }
  Ring rfreex;
  for (int64_t it = c.it0; it < a.npairs; it += c.itstep) {
    const int sd = c.side(a, it);
    const bool next = it + c.itstep < a.npairs;
    if (next) xn = next_points(false);
    if (ntc == 2) {
      // S_2 of this item, out of the accumulator: the values of the quads this warp will take
      wait(c.mid, midpar);
      midpar ^= 1;
      tc_fence_after();
      const int sn = next ? c.side(a, it + c.itstep) : 0;
      const float sc = c.steps[sd * 2].out_scale * c.steps[sd * 2 + 1].in_scale;
      const int nq = c.steps[sd * 2 + 1].nquads;
      float* s = s2;
      for (int q = first_quad(g + (next ? c.steps[sn * 2].nquads : 0)); q < nq; q += 4, s += 4 * TILE_M) {
        const float4 v = tmem_ld4(c.tmem + lanes + (uint32_t)(a.d2_col + 4 * q));
        s[0] = v.x * sc;
        s[TILE_M] = v.y * sc;
        s[2 * TILE_M] = v.z * sc;
        s[3 * TILE_M] = v.w * sc;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_cta0(c.d2free);
      if (next) {
        first_step(sn, xn[a.c1[sn]]);
        generate(sn, 0, s1, xn[c.steps[sn * 2].coord]);
      }
      generate(sd, 1, s2, xc[c.steps[sd * 2 + 1].coord]);
    } else {
      first_step(sd, xc[a.c1[sd]]);
      generate(sd, 0, s1, xc[c.steps[sd * 2].coord]);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&c.xempty[rfreex.slot]);
    rfreex.next(PAIR_XD);
    xc = xn;
  }
  if (dead && lane == 0) {
    *c.abort_flag = 1;
    atomicExch(a.status, (int)PTTK_ETIMEOUT);
  }
}

// 32 columns of this thread's row, scaled, into its staging row (cb + i < R only); R's largest power of
// two factor gives the width whose stores fall in distinct banks.
__device__ __forceinline__ void stage_row(float* dst, const float* v, float osc, int left, int width) {
  if (width == 1) {
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (i < left) dst[i] = v[i] * osc;
  } else if (width == 2) {
#pragma unroll
    for (int i = 0; i < 32; i += 2)
      if (i < left) *reinterpret_cast<float2*>(dst + i) = make_float2(v[i] * osc, v[i + 1] * osc);
  } else {
#pragma unroll
    for (int i = 0; i < 32; i += 4)
      if (i < left)
        *reinterpret_cast<float4*>(dst + i) = make_float4(v[i] * osc, v[i + 1] * osc, v[i + 2] * osc, v[i + 3] * osc);
  }
}

template <int FMT, bool SPLIT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PAIR_THREADS, 1) chain_pair_kernel(PairArgs a) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int np = a.np, np4 = np >> 2, ntc = a.ntc;
  const uint32_t na = (uint32_t)a.na, nb = (uint32_t)a.nb;
  PairCtx c;
  c.b_base = smem;                                                            // nb x b_slot
  c.stage = reinterpret_cast<float*>(c.b_base + (size_t)nb * a.b_slot);       // PAIR_EPI x 32 x stage_cols
  c.S1 = c.stage + (size_t)PAIR_EPI * 32 * a.stage_cols;                      // r1_pad x 128
  c.S2 = c.S1 + (size_t)a.r1_pad * TILE_M;                                    // s2_rows x 128
  c.G1 = c.S2 + (size_t)a.s2_rows * TILE_M;                                   // 2 x r1_pad x np
  c.X = c.G1 + (size_t)2 * a.r1_pad * np;                                     // PAIR_XD x 128 x d
  PairStep* steps = reinterpret_cast<PairStep*>(
      (reinterpret_cast<uintptr_t>(c.X + (size_t)PAIR_XD * TILE_M * a.d) + 15) & ~uintptr_t(15));  // [2][2]
  uint64_t* bars = reinterpret_cast<uint64_t*>(steps + 4);
  c.steps = steps;
  c.full_a = bars;
  c.full_b = bars + PAIR_MAX_NS;
  c.empty_a = bars + 2 * PAIR_MAX_NS;
  c.empty_b = bars + 3 * PAIR_MAX_NS;
  c.xfull = bars + 4 * PAIR_MAX_NS;
  c.xempty = c.xfull + PAIR_XD;
  c.mid = c.xempty + PAIR_XD;
  c.d2free = c.mid + 1;
  c.last_done = c.mid + 2;  // [2]
  c.rfree = c.mid + 4;      // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(c.mid + 6);
  c.abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  c.rank = cluster_rank();
  if (tid == 0) {
    for (uint32_t i = 0; i < na; ++i) {
      mbar_init(&c.full_a[i], 8);
      mbar_init(&c.empty_a[i], 1);
    }
    for (uint32_t i = 0; i < nb; ++i) {
      mbar_init(&c.full_b[i], c.rank == 0 ? 2 : 1);
      mbar_init(&c.empty_b[i], 1);
    }
    for (int i = 0; i < PAIR_XD; ++i) {
      mbar_init(&c.xfull[i], 32);
      mbar_init(&c.xempty[i], PAIR_GEN);
    }
    mbar_init(c.mid, 1);
    mbar_init(c.d2free, 2 * PAIR_GEN);
    for (int r = 0; r < 2; ++r) {
      mbar_init(&c.last_done[r], 1);
      mbar_init(&c.rfree[r], 2 * PAIR_EPI);
    }
    *c.abort_flag = 0;
    fence_mbar_init();
  }
  if (tid < 2 * ntc) steps[(tid / ntc) * 2 + tid % ntc] = a.st[tid / ntc][tid % ntc];
  for (int e = tid; e < 2 * a.r1_pad * np; e += PAIR_THREADS) {
    const int sd = e / (a.r1_pad * np), q = e % (a.r1_pad * np), o = q / np, j = q % np;
    c.G1[e] = (o < a.r1[sd] && j < a.n) ? a.g1[sd][j + a.n * o] : 0.f;
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  tc_fence_after();
  c.tmem = *tmem_slot;
  c.it0 = blockIdx.x >> 1;
  c.itstep = gridDim.x >> 1;
  const int64_t npairs = a.npairs;
  // The steps in the order in which every role works through them.
  auto for_steps = [&](auto&& step) {
    if (ntc == 2 && c.it0 < npairs && !step(c.side(a, c.it0), 0)) return;
    for (int64_t it = c.it0; it < npairs; it += c.itstep) {
      if (ntc == 2 && it + c.itstep < npairs && !step(c.side(a, it + c.itstep), 0)) return;
      if (!step(c.side(a, it), ntc - 1)) return;
    }
  };

  if (warp == 0) {
    // ---------------- core quads ----------------
    if (lane == 0) {
      Ring rb;
      bool ok = true;
      uint32_t used = 0;
      for_steps([&](int sd, int si) {
        const PairStep& st = steps[sd * 2 + si];
        const int nq = st.nquads;
        const uint32_t bytes = st.bytes;
        const uint8_t* src = st.img + (size_t)c.rank * bytes;
        for (int q = 0; q < nq; ++q, src += 2 * (size_t)bytes) {
          ok = mbar_wait(&c.empty_b[rb.slot], rb.par ^ 1, c.abort_flag);
          if (!ok) break;
          mbar_arrive_expect_tx(&c.full_b[rb.slot], bytes);
          tma_load_1d(c.b_base + (size_t)rb.slot * a.b_slot, src, bytes, &c.full_b[rb.slot]);
          rb.next(nb);
          used = used < nb ? used + 1 : nb;
        }
        return ok;
      });
      if (!ok) {
        *c.abort_flag = 1;
        atomicExch(a.status, (int)PTTK_ETIMEOUT);
      }
      // every copy has landed before the CTA ends: the last round of each slot, oldest first
      const int zero = 0;
      for (uint32_t k = used; k > 0; --k) {
        const bool back = rb.slot < k;
        mbar_wait(&c.full_b[back ? rb.slot + nb - k : rb.slot - k], back ? rb.par ^ 1 : rb.par, &zero);
      }
    }
    __syncwarp();
  } else if (warp == 1 && c.rank == 1) {
    // ---------------- CTA 1: its core quads' arrival, passed on to CTA 0 ----------------
    if (lane == 0) {
      Ring rb;
      bool ok = true;
      for_steps([&](int sd, int si) {
        for (int q = 0, nq = steps[sd * 2 + si].nquads; q < nq && ok; ++q) {
          ok = mbar_wait(&c.full_b[rb.slot], rb.par, c.abort_flag);
          if (ok) arrive_cta0(&c.full_b[rb.slot]);
          rb.next(nb);
        }
        return ok;
      });
      if (!ok) {
        *c.abort_flag = 1;
        atomicExch(a.status, (int)PTTK_ETIMEOUT);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- CTA 0: MMAs of the pair ----------------
    const bool lead = elect_one();
    Ring ra, rb, rd;         // A slots, core slots, output accumulators
    uint32_t d2par = 0, first = 1, prev = 0, prev_par = 0;
    bool ok = true, any = false;
    const uint32_t tmem = __shfl_sync(0xffffffffu, c.tmem, 0);
    const uint32_t sbase = __shfl_sync(0xffffffffu, smem_u32(c.b_base), 0);
    const uint32_t sbo = 64u * (uint32_t)np;  // 8-row group stride of a core quad
    for_steps([&](int sd, int si) {
      const PairStep& st = a.st[sd][si];
      const uint32_t idesc = st.idesc, idesc_neg = st.idesc | (1u << 13);  // bit 13: negate A
      const uint32_t lo_off = st.bytes >> 5;
      const int nq = st.nquads;
      const bool last = si == ntc - 1;
      uint32_t dacc;
      uint64_t* done;
      if (!last) {
        // the previous item's S_2 has been read out of the accumulator
        if (!first) {
          ok = mbar_wait(c.d2free, d2par, c.abort_flag);
          d2par ^= 1;
        }
        first = 0;
        dacc = tmem + (uint32_t)a.d2_col;
        done = c.mid;
      } else {
        ok = mbar_wait(&c.rfree[rd.slot], rd.par ^ 1, c.abort_flag);
        dacc = tmem + rd.slot * (uint32_t)a.d_cols;
        done = &c.last_done[rd.slot];
        rd.next((uint32_t)a.nd);
      }
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) return false;
      tc_fence_after();
      for (int q = 0; q < nq; ++q) {
        ok = mbar_wait(&c.full_b[rb.slot], rb.par, c.abort_flag) && mbar_wait(&c.full_a[ra.slot], ra.par, c.abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return false;
        tc_fence_after();
        const uint32_t ta = tmem + (uint32_t)(a.a_col) + ra.slot * (uint32_t)a.slot_cols;
        const uint64_t b0 = smem_desc2(sbase + rb.slot * a.b_slot, sbo);
        if (lead) {
          for (int k = 0; k < np4; ++k) {
            const uint64_t bh = b0 + (uint64_t)(16 * k);
            pair_umma(dacc, ta + 8 * k, bh, idesc, (q > 0 || k > 0) ? 1u : 0u);
            if (SPLIT) {
              pair_umma(dacc, ta + 8 * k, bh + lo_off, idesc, 1u);
              pair_umma(dacc, ta + 2 * np + 8 * k, bh, idesc_neg, 1u);
            }
          }
          pair_commit(&c.empty_a[ra.slot]);
          pair_commit(&c.empty_b[rb.slot]);
          if (q == nq - 1) pair_commit(done);
        }
        __syncwarp();
        prev = ra.slot;
        prev_par = ra.par;
        any = true;
        ra.next(na);
        rb.next(nb);
      }
      return true;
    });
    if (!ok && lane == 0) {
      *c.abort_flag = 1;
      atomicExch(a.status, (int)PTTK_ETIMEOUT);
    }
    const int zero = 0;
    if (any) mbar_wait(&c.empty_a[prev], prev_par, &zero);
    __syncwarp();
  } else if (warp == 3) {
    // ---------------- points: 128 rows x d per item, rows past the end read as the last row ----------------
    Ring rx;
    bool ok = true;
    const int d = a.d;
    for (int64_t it = c.it0; it < npairs; it += c.itstep) {
      const int sd = c.side(a, it);
      ok = mbar_wait(&c.xempty[rx.slot], rx.par ^ 1, c.abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const int64_t row0 = c.row0(a, it), lastrow = a.N[sd] - 1;
      const float* src = a.pts[sd];
      const uint32_t dst = smem_u32(c.X + (size_t)rx.slot * TILE_M * d);
      for (int e = lane; e < TILE_M * d; e += 32) {
        const int r = d == 3 ? (e * 43691) >> 17 : e >> 1;  // e / d for d = 3 (e < 384) or 2
        const int64_t p = std::min<int64_t>(row0 + r, lastrow);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * (uint32_t)e), "l"(src + p * d + (e - r * d))
                     : "memory");
      }
      asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&c.xfull[rx.slot])) : "memory");
      rx.next(PAIR_XD);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok && lane == 0) {
      *c.abort_flag = 1;
      atomicExch(a.status, (int)PTTK_ETIMEOUT);
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 4 + PAIR_GEN) {
    // ---------------- generators ----------------
    switch (np4) {
      case 1: pair_generate<FMT, SPLIT, 4>(a, c); break;
      case 2: pair_generate<FMT, SPLIT, 8>(a, c); break;
      case 3: pair_generate<FMT, SPLIT, 12>(a, c); break;
      case 4: pair_generate<FMT, SPLIT, 16>(a, c); break;
      case 5: pair_generate<FMT, SPLIT, 20>(a, c); break;
      case 6: pair_generate<FMT, SPLIT, 24>(a, c); break;
      case 7: pair_generate<FMT, SPLIT, 28>(a, c); break;
      default: pair_generate<FMT, SPLIT, 32>(a, c); break;
    }
  } else if (warp >= 4 + PAIR_GEN) {
    // ---------------- output: one warp per lane quarter ----------------
    const int quarter = warp & 3;
    const uint32_t lanes = (uint32_t)(32 * quarter) << 16;
    float* stg = c.stage + (size_t)quarter * 32 * a.stage_cols;
    Ring rd;
    bool dead = false;
    for (int64_t it = c.it0; it < npairs; it += c.itstep) {
      const int sd = c.side(a, it);
      const PairStep& st = steps[sd * 2 + ntc - 1];
      if (!dead) dead = !mbar_wait(&c.last_done[rd.slot], rd.par, c.abort_flag);
      dead = __any_sync(0xffffffffu, dead);
      // the previous item's copy has read the staging rows
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
      tc_fence_after();
      const int R = st.R_out;
      const int64_t row0 = c.row0(a, it) + 32 * quarter;
      const int wrows = (int)std::max<int64_t>(0, std::min<int64_t>(32, a.N[sd] - row0));
      if (!dead) {
        const int width = R & 1 ? 1 : R & 2 ? 2 : 4;
        for (int cb = 0; cb < R; cb += 32) {
          float v[32];
          tmem_ld32_wait(c.tmem + lanes + rd.slot * (uint32_t)a.d_cols + (uint32_t)cb, v);
          stage_row(stg + (size_t)lane * R + cb, v, st.out_scale, R - cb, width);
        }
      }
      tc_fence_before();
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) arrive_cta0(&c.rfree[rd.slot]);
      rd.next((uint32_t)a.nd);
      if (!dead && wrows > 0) {
        float* out = a.out[sd] + row0 * R;
        if (wrows == 32 && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
          if (lane == 0) {
            asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(out), "r"(smem_u32(stg)),
                         "r"((uint32_t)(32 * R * 4))
                         : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        } else {
          for (int e = lane; e < wrows * R; e += 32) out[e] = stg[e];
        }
        __syncwarp();
      }
    }
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (dead && lane == 0) {
      *c.abort_flag = 1;
      atomicExch(a.status, (int)PTTK_ETIMEOUT);
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' work on either tensor memory and every remote arrival is over
  tc_fence_after();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(c.tmem) : "memory");
  cluster_sync_all();
}

// Image of an oriented core (K x R_out, column-major, FP64; K = n R_in) in the order above: quad c
// holds the values a = 4 c .. 4 c + 3, first CTA 0's Npad / 2 columns, then CTA 1's, each the high
// parts and then the residuals, K-major without swizzle (16-byte units of 8 values of K, core matrices of 8 rows, row groups 64 np
// bytes apart).
template <int FMT>
__global__ void pair_image_kernel(const double* __restrict__ G, int n, int np, int R_in, int R_out, int Npad,
                                  int nquads, bool split, double scale, uint8_t* __restrict__ img) {
  const int KC = 4 * np, Nh = Npad / 2;
  const size_t part = (size_t)Nh * KC * 2, quad = part * (split ? 2 : 1);
  const int64_t total = (int64_t)nquads * Npad * KC;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int kk = (int)(e % KC), o = (int)((e / KC) % Npad), c = (int)(e / ((int64_t)KC * Npad));
    const int ai = 4 * c + kk / np, j = kk % np;
    const double v = (ai < R_in && j < n && o < R_out) ? scale * G[(ai + R_in * j) + (int64_t)n * R_in * o] : 0.0;
    const int cta = o / Nh, ro = o % Nh;
    uint8_t* hi = img + ((size_t)c * 2 + cta) * quad + (size_t)(ro >> 3) * (64 * np) + (size_t)(kk >> 3) * 128 +
                  (size_t)(ro & 7) * 16 + (size_t)(kk & 7) * 2;
    if constexpr (FMT == FMT_BF16) {
      const __nv_bfloat16 h = __double2bfloat16(v);
      *reinterpret_cast<__nv_bfloat16*>(hi) = h;
      if (split) *reinterpret_cast<__nv_bfloat16*>(hi + part) = __double2bfloat16(v - (double)__bfloat162float(h));
    } else {
      const __half h = __double2half(v);
      *reinterpret_cast<__half*>(hi) = h;
      if (split) *reinterpret_cast<__half*>(hi + part) = __double2half(v - (double)__half2float(h));
    }
  }
}

bool pair_split(pttk_prec p) { return p == PTTK_BF16X3 || p == PTTK_FP16X3; }
bool pair_bf16(pttk_prec p) { return p == PTTK_BF16 || p == PTTK_BF16X3; }

// Launch arguments that depend on the handle and the form alone; false where the kernel cannot
// hold the ranks (the caller's other kernels then take the call).
bool pair_plan(const pttk_tt* tt, pttk_prec prec, PairArgs& a, size_t* smem_out) {
  const int parts = pair_split(prec) ? 2 : 1;
  a = PairArgs{};
  a.n = tt->n;
  a.d = tt->d;
  a.np = (tt->n + 3) / 4 * 4;
  a.ntc = tt->d - 1;
  int npad_last = 16, npad_mid = 0;
  for (int side = 0; side < 2; ++side) {
    int rin, rout, coord;
    oriented_core_dims(tt, side == 0, 0, &rin, &rout, &coord);
    if (rin != 1) return false;
    a.r1[side] = rout;
    a.c1[side] = coord;
    a.r1_pad = std::max(a.r1_pad, (rout + 15) / 16 * 16);
    const int b1 = side == 0 ? coord : tt->d + tt->dtheta + coord;
    a.lo1[side] = (float)tt->box[b1][0];
    a.hi1[side] = (float)tt->box[b1][1];
    for (int i = 0; i < a.ntc; ++i) {
      PairStep& st = a.st[side][i];
      oriented_core_dims(tt, side == 0, i + 1, &rin, &rout, &coord);
      st.nquads = (rin + 3) / 4;
      st.R_out = rout;
      st.Npad = (rout + 15) / 16 * 16;
      if (st.Npad > 256) return false;
      st.bytes = (uint32_t)(parts * (st.Npad / 2) * 4 * a.np * 2);
      st.idesc = instr_desc(pair_bf16(prec) ? fmt_code(FMT_BF16) : fmt_code(FMT_FP16), 256, st.Npad);
      st.coord = coord;
      const int bj = side == 0 ? coord : tt->d + tt->dtheta + coord;
      st.lo = (float)tt->box[bj][0];
      st.hi = (float)tt->box[bj][1];
      a.b_slot = std::max(a.b_slot, st.bytes);
      if (i == a.ntc - 1) {
        npad_last = std::max(npad_last, st.Npad);
        a.stage_cols = std::max(a.stage_cols, (rout + 3) / 4 * 4);
      }
      else npad_mid = std::max(npad_mid, st.Npad);
    }
  }
  a.s2_rows = npad_mid;
  a.d_cols = (npad_last + 31) / 32 * 32;
  const int mid_cols = (npad_mid + 31) / 32 * 32;
  const int quad_cols = parts * 2 * a.np;
  // two output accumulators where they leave room for four quads of A, else one (its readout then
  // runs behind the next item's first tensor-core step)
  a.nd = 2 * a.d_cols + mid_cols + 4 * quad_cols <= 512 ? 2 : 1;
  a.slot_cols = quad_cols;
  a.d2_col = a.nd * a.d_cols;
  a.a_col = a.d2_col + mid_cols;
  const size_t fixed = sizeof(float) * ((size_t)PAIR_EPI * 32 * a.stage_cols + (size_t)a.r1_pad * TILE_M +
                                        (size_t)a.s2_rows * TILE_M + (size_t)2 * a.r1_pad * a.np + (size_t)PAIR_XD * TILE_M * a.d) +
                       16 + 4 * sizeof(PairStep) + 8 * (4 * PAIR_MAX_NS + 2 * PAIR_XD + 6) + 16;
  const size_t limit = 227 * 1024;
  if (a.a_col >= 512 || fixed >= limit) return false;
  a.na = std::min(PAIR_MAX_NS, (512 - a.a_col) / a.slot_cols);
  a.b_slot = (a.b_slot + 127) / 128 * 128;
  a.nb = std::min<int>(PAIR_MAX_NS, (int)((limit - fixed) / a.b_slot));
  // a warp's quads are four apart, so with four slots the one it waits on is never two rounds behind
  // (a parity wait cannot tell rounds two apart)
  if (a.na < 4 || a.nb < 3) return false;
  *smem_out = std::max<size_t>((size_t)a.nb * a.b_slot + fixed, 116 * 1024);  // one CTA (one TMEM allocation) per SM
  return true;
}

template <int FMT, bool SPLIT>
pttk_status launch_pair(const PairArgs& a, size_t smem, cudaStream_t s) {
  auto kfn = chain_pair_kernel<FMT, SPLIT>;
  PTTK_CUDA(allow_smem((const void*)kfn));
  const int64_t clusters = std::max<int64_t>(1, std::min<int64_t>(a.npairs, sm_count() / 2));
  kfn<<<(unsigned)(2 * clusters), PAIR_THREADS, smem, s>>>(a);
  pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

}  // namespace

bool pair_form(const pttk_tt* tt, pttk_prec prec) {
  if (tt->d < 2 || !(prec == PTTK_FP16 || prec == PTTK_FP16X3 || pair_bf16(prec))) return false;
  PairArgs a;
  size_t smem;
  return pair_plan(tt, prec, a, &smem);
}

// Images and the powers of two of the FP16 forms: image scale 2^sB with max|G| 2^sB <= 2^14,
// and S_in of each step stored times 2^sA with bound(|S_in|) 2^sA <= 2^14, where
// bound(S_1) = the largest column 1-norm of the first core and bound(S_out) = bound(S_in) times that
// of the step's core (|T_j| <= 1).
pttk_status pair_prepare(const pttk_tt* tt, pttk_prec prec, PairImages& im, cudaStream_t s) {
  PairArgs a;
  size_t smem;
  if (!pair_plan(tt, prec, a, &smem)) return set_error(PTTK_ENOTSUP, "pair chain: ranks do not fit");
  const bool bf16 = pair_bf16(prec), split = pair_split(prec);
  size_t total = 0;
  for (int side = 0; side < 2; ++side)
    for (int i = 0; i < a.ntc; ++i) {
      im.off[side][i] = total;
      total += (size_t)a.st[side][i].nquads * 2 * a.st[side][i].bytes;
    }
  uint8_t* buf = nullptr;
  PTTK_CUDA(cudaMalloc(&buf, std::max<size_t>(total, 16)));
  auto body = [&]() -> pttk_status {
    for (int side = 0; side < 2; ++side) {
      double bound = 1.0;
      for (int i = -1; i < a.ntc; ++i) {
        int rin, rout, coord;
        const int k = oriented_core_dims(tt, side == 0, i + 1, &rin, &rout, &coord);
        const double* G = static_cast<const double*>(oriented_core_ptr(tt, side == 0, k, true));
        double img_scale = 1.0;
        if (!bf16) {
          const int64_t K = (int64_t)tt->n * rin;
          std::vector<double> h((size_t)(K * rout));
          PTTK_CUDA(cudaMemcpyAsync(h.data(), G, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, s));
          PTTK_CUDA(cudaStreamSynchronize(s));
          double gmax = 0.0, colmax = 0.0;
          for (int o = 0; o < rout; ++o) {
            double sum = 0.0;
            for (int64_t q = 0; q < K; ++q) {
              const double g = fabs(h[(size_t)(q + K * o)]);
              gmax = std::max(gmax, g);
              sum += g;
            }
            colmax = std::max(colmax, sum);
          }
          if (i >= 0) {
            const int sB = gmax > 0.0 ? 14 - (int)ceil(log2(gmax)) : 0;
            const int sA = bound > 0.0 ? 14 - (int)ceil(log2(bound)) : 0;
            img_scale = ldexp(1.0, sB);
            im.in_scale[side][i] = (float)ldexp(1.0, sA);
            im.out_scale[side][i] = (float)ldexp(1.0, -(sA + sB));
          }
          bound *= std::max(colmax, 1e-300);
        } else if (i >= 0) {
          im.in_scale[side][i] = im.out_scale[side][i] = 1.f;
        }
        if (i < 0) continue;
        const PairStep& st = a.st[side][i];
        const int64_t work = (int64_t)st.nquads * st.Npad * 4 * a.np;
        const unsigned blocks = (unsigned)std::min<int64_t>((work + 255) / 256, (int64_t)sm_count() * 8);
        auto* kfn = bf16 ? pair_image_kernel<FMT_BF16> : pair_image_kernel<FMT_FP16>;
        kfn<<<blocks, 256, 0, s>>>(G, tt->n, a.np, rin, rout, st.Npad, st.nquads, split, img_scale, buf + im.off[side][i]);
        pttk::count_launch();
      }
    }
    PTTK_CUDA(cudaGetLastError());
    PTTK_CUDA(cudaStreamSynchronize(s));
    return PTTK_OK;
  };
  const pttk_status st = body();
  if (st != PTTK_OK) {
    cudaFree(buf);
    return st;
  }
  im.buf = buf;
  return PTTK_OK;
}

pttk_status pair_build(const pttk_tt* tt, pttk_prec prec, const PairImages& im, const float* X, int64_t N_s,
                       const float* Y, int64_t N_t, float* U, float* V, int* d_status, cudaStream_t s) {
  PairArgs a;
  size_t smem;
  if (!pair_plan(tt, prec, a, &smem)) return set_error(PTTK_ENOTSUP, "pair chain: ranks do not fit");
  for (int side = 0; side < 2; ++side) {
    int rin, rout, coord;
    const int k = oriented_core_dims(tt, side == 0, 0, &rin, &rout, &coord);
    a.g1[side] = static_cast<const float*>(oriented_core_ptr(tt, side == 0, k, false));
    for (int i = 0; i < a.ntc; ++i) {
      a.st[side][i].img = im.buf + im.off[side][i];
      a.st[side][i].in_scale = im.in_scale[side][i];
      a.st[side][i].out_scale = im.out_scale[side][i];
    }
  }
  a.N[0] = N_s;
  a.N[1] = N_t;
  a.P0 = (N_s + 2 * TILE_M - 1) / (2 * TILE_M);
  a.npairs = a.P0 + (N_t + 2 * TILE_M - 1) / (2 * TILE_M);
  a.pts[0] = X;
  a.pts[1] = Y;
  a.out[0] = U;
  a.out[1] = V;
  a.status = d_status;
  PTTK_PROF("chain_tc", s);
  if (pair_bf16(prec))
    return pair_split(prec) ? launch_pair<FMT_BF16, true>(a, smem, s) : launch_pair<FMT_BF16, false>(a, smem, s);
  return pair_split(prec) ? launch_pair<FMT_FP16, true>(a, smem, s) : launch_pair<FMT_FP16, false>(a, smem, s);
}

}  // namespace pttk
