// Online stage: H(theta) (Eq. hmat, Algorithm 3), the factor chains of Algorithm 2,
// Phase 3 (SIMT FP64 / FP32 form), and the low-rank product U (M (V^T w)).
//
// Factor chain. Per point p the source chain is
//   S_1 = B_1 G_1^{2},   S_i = (B_i face-split S_{i-1}) G_i^{2},   U[p, :] = S_d,
// with B_i[p, k] = T_k(xhat_{p,i}) and the Kronecker column index a + r_{i-1} j matching
// the row index of G_i^{2}. The target chain T <- G_D^{1} V_d^T,
// T <- G_{D-i}^{1} (T Khatri-Rao V_{d-i}^T) has the same per-point form once each core is
// read as (input rank, j, output rank) = (right rank, j, left rank); the handle keeps those
// transposed copies of the target-side cores ("oriented" cores). Each chain step is then a
// GEMM  S_out (P x R_out) = A (P x n R_in) * Gs^{2} (n R_in x R_out)  whose A operand
// A[p, a + R_in j] = B[p, j] S_in[p, a] is generated in shared memory, never stored.
#include <math.h>

#include <stdio.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <mutex>
#include <type_traits>

#include "pttk_internal.cuh"

namespace pttk {

int oriented_core_dims(const pttk_tt* tt, bool source, int step, int* R_in, int* R_out,
                       int* coord);

namespace {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <typename T>
__device__ __forceinline__ T warp_sum(T v);
template <>
__device__ __forceinline__ double warp_sum<double>(double v) { return warp_sum_d(v); }
template <>
__device__ __forceinline__ float warp_sum<float>(float v) { return warp_sum_f(v); }

// ---------------- H(theta) -------------------------------------------------------------
// One or two theta cores contracted with their Chebyshev vectors in one launch (blockIdx.y: the core), G
// (ra x n x rb, column-major): sum_k G[a + ra (k + n b)] T_k(th), into out[a + ra b], or, for a single core, row-major
// into M.
struct ThetaCores {
  const double* G[2];
  double* out[2];
  double th[2];
  int ra[2], rb[2];
};
template <typename T>
__global__ void __launch_bounds__(256) contract_theta_kernel(ThetaCores c, int n, T* __restrict__ M) {
  const int q = blockIdx.y;
  const double* __restrict__ G = c.G[q];
  const int ra = c.ra[q], rb = c.rb[q];
  const double th = c.th[q];
  const int64_t total = (int64_t)ra * rb;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int a = (int)(e % ra), b = (int)(e / ra);
    const double* g = G + a + (int64_t)ra * n * b;
    double t0 = 1.0, t1 = th, acc = 0.0;
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
      acc = fma(g[(int64_t)ra * k], t0, acc);
      const double t2 = 2.0 * th * t1 - t0;
      t0 = t1;
      t1 = t2;
    }
    if (M) M[(int64_t)a * rb + b] = (T)acc;
    else c.out[q][e] = acc;
  }
}

// H = H1 H2 for two theta cores, split over the inner dimension so that the product spreads
// over the whole GPU (FP64 issue is ~2 DFMA per clock per SM here, so a few output tiles on a
// few SMs would take ~0.5 ms): block (tile, slice) writes
//   part[slice][a + rs b] = sum_{c in slice} H1[a + rs c] H2[c + rm b]
// and hprod_reduce_kernel sums the slices in a fixed order.
constexpr int HP_T = 32;  // output tile edge and inner slice length
__global__ void __launch_bounds__(256) hprod_splitk_kernel(const double* __restrict__ H1,
                                                           const double* __restrict__ H2, int rs,
                                                           int rm, int rt,
                                                           double* __restrict__ part) {
  __shared__ double a_s[HP_T][HP_T + 1], b_s[HP_T][HP_T + 1];
  const int a0 = blockIdx.x * HP_T, b0 = blockIdx.y * HP_T, c0 = blockIdx.z * HP_T;
  for (int e = threadIdx.x; e < HP_T * HP_T; e += blockDim.x) {
    const int i = e % HP_T, j = e / HP_T;  // a_s[i][j] = H1[a0 + i, c0 + j]; b_s[i][j] = H2[c0 + i, b0 + j]
    a_s[i][j] = (a0 + i < rs && c0 + j < rm) ? H1[(a0 + i) + (int64_t)rs * (c0 + j)] : 0.0;
    b_s[i][j] = (c0 + i < rm && b0 + j < rt) ? H2[(c0 + i) + (int64_t)rm * (b0 + j)] : 0.0;
  }
  __syncthreads();
  const int ti = threadIdx.x % HP_T, tj = threadIdx.x / HP_T;  // tj in [0, 8)
  double acc[HP_T / 8] = {};
  for (int c = 0; c < HP_T; ++c) {
    const double av = a_s[ti][c];
#pragma unroll
    for (int q = 0; q < HP_T / 8; ++q) acc[q] = fma(av, b_s[c][tj + 8 * q], acc[q]);
  }
  double* out = part + (int64_t)blockIdx.z * rs * rt;
#pragma unroll
  for (int q = 0; q < HP_T / 8; ++q) {
    const int a = a0 + ti, b = b0 + tj + 8 * q;
    if (a < rs && b < rt) out[a + (int64_t)rs * b] = acc[q];
  }
}

// M row-major (rs x rt) = sum over the slices of part, in slice order
template <typename T>
__global__ void hprod_reduce_kernel(const double* __restrict__ part, int nslices, int rs, int rt,
                                    T* __restrict__ M) {
  const int64_t total = (int64_t)rs * rt;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = e / rt, b = e % rt;
    double acc = 0.0;
    for (int sl = 0; sl < nslices; ++sl) acc += part[(int64_t)sl * total + a + (int64_t)rs * b];
    M[e] = (T)acc;
  }
}

__global__ void identity_rowmajor_kernel(void* M, int r, bool fp64) {
  const int64_t total = (int64_t)r * r;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const double v = (e / r == e % r) ? 1.0 : 0.0;
    if (fp64) static_cast<double*>(M)[e] = v;
    else static_cast<float*>(M)[e] = (float)v;
  }
}

// ---------------- factor chain (SIMT) -----------------------------------------------
struct ChainStep {
  const void* G;  // oriented core, column-major (R_in x n x R_out)
  int R_in, R_out, coord, ct;  // ct: output columns per pass (0: the narrow form)
  uint32_t magic;              // ceil(2^32 / R_in): k / R_in = umulhi(k, magic) (R_in > 1)
  double lo, hi;
};
struct ChainSide {
  ChainStep st[3];
  const void* pts;
  void* out;
  int64_t N;
};
struct ChainArgs {
  ChainSide side[2];
  int nsteps, n, d;
  int64_t blocks0;  // blocks of side 0
  int rin_max;      // largest R_in of a step
};

constexpr int BK = 16;      // values of K per chunk
constexpr int NARROW = 16;  // steps of at most this many outputs take the narrow form

__device__ __forceinline__ void fma_pair(double a, const double* b, double* acc) {
  acc[0] = fma(a, b[0], acc[0]);
  acc[1] = fma(a, b[1], acc[1]);
}
__device__ __forceinline__ void fma_pair(float a, const float* b, float* acc) {
  // the two-wide FP32 FMA: each half rounds as fmaf does
  uint64_t x, y, z;
  asm("mov.b64 %0, {%1, %1};" : "=l"(x) : "f"(a));
  asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b[0]), "f"(b[1]));
  asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(acc[0]), "f"(acc[1]));
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(z) : "l"(x), "l"(y), "l"(z));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[0]), "=f"(acc[1]) : "l"(z));
}

// One chain step of a block's P = 16 TM points: 16 x 16 threads, each TM points x TN outputs (the pairs
// 32 jj + 2 tx, + 1), CT = 16 TN outputs per pass. A[k][p] = T_j S_in[a] is formed chunk by chunk in
// shared memory beside the core's chunk, which was loaded one chunk ahead into registers; the two chunk
// buffers alternate, so a chunk costs one barrier. Every output is summed over k in order.
template <typename T, int TM, int TN>
__device__ void chain_step(const ChainStep& st, int n, const T* __restrict__ Bv, const T* __restrict__ Sin,
                           T* __restrict__ Sout, T* __restrict__ As, T* __restrict__ Gs, T* __restrict__ out, int64_t p0,
                           int64_t N, bool last) {
  constexpr int P = 16 * TM, CT = 16 * TN, GL = CT + 2;
  constexpr int NA = BK * P / 256, NG = BK * CT / 256;
  const T* __restrict__ G = static_cast<const T*>(st.G);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int K = n * st.R_in;
  for (int o0 = 0; o0 < st.R_out; o0 += CT) {
    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[i][j] = T(0);
    T greg[NG];
    auto load_g = [&](int k0) {
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const int e = tid + 256 * i, kk = e % BK, o = e / BK;
        greg[i] = (k0 + kk < K && o0 + o < st.R_out) ? __ldg(G + (k0 + kk) + (int64_t)K * (o0 + o)) : T(0);
      }
    };
    load_g(0);
    int buf = 0;
    for (int k0 = 0; k0 < K; k0 += BK, buf ^= 1) {
      T* Ab = As + buf * BK * P;
      T* Gb = Gs + buf * BK * GL;
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const int e = tid + 256 * i;
        Gb[(e % BK) * GL + e / BK] = greg[i];
      }
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int e = tid + 256 * i, kk = e / P, p = e % P, k = k0 + kk;
        T v = T(0);
        if (k < K) {
          const int j = st.R_in > 1 ? (int)__umulhi((uint32_t)k, st.magic) : k;
          v = Bv[j * P + p] * Sin[(k - j * st.R_in) * P + p];
        }
        Ab[kk * P + p] = v;
      }
      __syncthreads();
      if (k0 + BK < K) load_g(k0 + BK);
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        T av[TM], bv[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) av[i] = Ab[kk * P + ty * TM + i];
#pragma unroll
        for (int j = 0; j < TN; j += 2) {
          bv[j] = Gb[kk * GL + 16 * j + 2 * tx];
          bv[j + 1] = Gb[kk * GL + 16 * j + 2 * tx + 1];
        }
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; j += 2) fma_pair(av[i], bv + j, acc[i] + j);
      }
    }
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int oc = o0 + 16 * (j & ~1) + 2 * tx + (j & 1);
      if (oc >= st.R_out) continue;
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const int p = ty * TM + i;
        if (last) {
          if (p0 + p < N) out[(p0 + p) * st.R_out + oc] = acc[i][j];
        } else {
          Sout[oc * P + p] = acc[i][j];
        }
      }
    }
    __syncthreads();  // the chunk buffers are free again, and S_out is complete after the last pass
  }
}

// A step of at most NARROW outputs: one output per thread at a time, the core's values read as
// broadcasts. In the tiled form a first step (n values of K, about 10 outputs) would compute 64 columns: 10 %
// of a d = 2 chain.
template <typename T, int P>
__device__ void chain_step_narrow(const ChainStep& st, int n, const T* __restrict__ Bv, const T* __restrict__ Sin,
                                  T* __restrict__ Sout, T* __restrict__ out, int64_t p0, int64_t N, bool last) {
  const T* __restrict__ G = static_cast<const T*>(st.G);
  const int K = n * st.R_in;
  for (int e = threadIdx.x; e < P * st.R_out; e += 256) {
    const int p = e % P, o = e / P;
    T acc = T(0);
    for (int j = 0, k = 0; j < n; ++j) {
      const T b = Bv[j * P + p];
      for (int ar = 0; ar < st.R_in; ++ar, ++k) acc = fma(b * Sin[ar * P + p], __ldg(G + k + (int64_t)K * o), acc);
    }
    if (!last) Sout[o * P + p] = acc;
    else if (p0 + p < N) out[(p0 + p) * st.R_out + o] = acc;
  }
  __syncthreads();
}

// Factor rows of both sides: a block takes 16 TM points of one side. TM is chosen by the point counts and
// ranks (factor_build_run). What bounds it: FMA issue. 200k points a side, ranks 10, 63 | 63, 12, n = 20:
// FP32 1.156 -> 0.38 ms, FP64 11.13 -> 9.95 ms (9.05 ms at the DFMA rate), against 64 points x 64 columns a
// block, 4 x 4 a thread, one buffer and a tiled first step.
// CTMAX, the widest pass any step takes, sets the registers: FP32 up to 64 columns runs three blocks an SM (two:
// 0.457 ms), all others two (FP64 with one: 10.25 ms).
template <typename T, int TM, int CTMAX>
__global__ void __launch_bounds__(256, sizeof(T) == 4 && CTMAX == 64 ? 3 : 2) chain_kernel(ChainArgs a) {
  constexpr int P = 16 * TM;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int sd = (int64_t)blockIdx.x < a.blocks0 ? 0 : 1;
  const ChainSide& side = a.side[sd];
  const int n = a.n;
  T* Sin = reinterpret_cast<T*>(smem_raw);      // rin_max x P
  T* Sout = Sin + (size_t)a.rin_max * P;
  T* Bv = Sout + (size_t)a.rin_max * P;         // n x P basis values
  T* As = Bv + (size_t)n * P;                   // 2 x BK x P
  T* Gs = As + 2 * BK * P;                      // 2 x BK x (ct + 2): the transposed stores of a core chunk meet the fewest bank conflicts
  const int64_t p0 = ((int64_t)blockIdx.x - (sd ? a.blocks0 : 0)) * P, N = side.N;
  const T* __restrict__ pts = static_cast<const T*>(side.pts);
  T* out = static_cast<T*>(side.out);
  // S_0 = 1 (r_0 = 1)
  for (int p = threadIdx.x; p < P; p += 256) Sin[p] = T(1);
  for (int si = 0; si < a.nsteps; ++si) {
    const ChainStep& st = side.st[si];
    // Chebyshev basis of this coordinate by the three-term recurrence
    for (int p = threadIdx.x; p < P; p += 256) {
      const int64_t gp = p0 + p;
      const T x = gp < N ? pts[gp * a.d + st.coord] : T(st.lo);
      const T xh = (T(2) * x - T(st.lo) - T(st.hi)) / (T(st.lo) - T(st.hi));
      T t0 = T(1), t1 = xh;
      Bv[p] = t0;
      if (n > 1) Bv[P + p] = t1;
      for (int k = 2; k < n; ++k) {
        const T t2 = T(2) * xh * t1 - t0;
        Bv[k * P + p] = t2;
        t0 = t1;
        t1 = t2;
      }
    }
    __syncthreads();
    const bool last = si == a.nsteps - 1;
    switch (st.ct) {
      case 0: chain_step_narrow<T, P>(st, n, Bv, Sin, Sout, out, p0, N, last); break;
      case 64: chain_step<T, TM, 4>(st, n, Bv, Sin, Sout, As, Gs, out, p0, N, last); break;
      case 96: if constexpr (CTMAX >= 96) chain_step<T, TM, 6>(st, n, Bv, Sin, Sout, As, Gs, out, p0, N, last); break;
      default: if constexpr (CTMAX >= 128) chain_step<T, TM, 8>(st, n, Bv, Sin, Sout, As, Gs, out, p0, N, last); break;
    }
    T* tmp = Sin;
    Sin = Sout;
    Sout = tmp;
  }
}

// ---------------- apply: out = U (M (V^T w)) ----------------------------------------
// partial[b, c] = sum over block b's rows r of V[r, c] w[r], in one of two forms (apply_typed chooses).
//
// By columns: threads are 4 row lanes x 64 columns, four rows of loads in flight each.
template <typename T>
__global__ void __launch_bounds__(256) vtw_columns_kernel(const T* __restrict__ V, int64_t N, int rt,
                                                          const T* __restrict__ w, T* __restrict__ partial) {
  __shared__ T red[4][64];
  const int64_t per = (N + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = (int64_t)blockIdx.x * per, r1 = std::min<int64_t>(N, r0 + per);
  const int cl = threadIdx.x & 63, rl = threadIdx.x >> 6;
  for (int cb = 0; cb < rt; cb += 64) {
    const int c = cb + cl;
    const bool on = c < rt;
    T acc[1] = {T(0)};
    int64_t r = r0 + rl;
    for (; r + 12 < r1; r += 16) {
      T v[4][1];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const T* src = V + (r + 4 * u) * rt + c;
        v[u][0] = on ? *src : T(0);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const T wr = w[r + 4 * u];
        acc[0] = fma(v[u][0], wr, acc[0]);
      }
    }
    for (; r < r1; r += 4) {
      const T wr = w[r];
      acc[0] = fma(on ? V[r * rt + c] : T(0), wr, acc[0]);
    }
    red[rl][cl] = acc[0];
    __syncthreads();
    for (int q = threadIdx.x; q < 64; q += blockDim.x)
      if (cb + q < rt) partial[(int64_t)blockIdx.x * rt + cb + q] = (red[0][q] + red[1][q]) + (red[2][q] + red[3][q]);
    __syncthreads();
  }
}

// Flat: V as an array of 16-byte units (of VW elements, whatever rt is): a unit of P rows (P rt a multiple of VW)
// always covers the same columns, so thread t keeps accumulators whose columns and row offsets never change (VW for
// each of the UNR groups in flight, so that no sum is a longer chain than in the form above), and takes unit t of
// every group of P rows; nt = P rt / VW threads make a group, and as many groups as fit run side by side. The
// accumulators of a column meet in shared memory in a fixed order.
template <typename T, int VW>
__global__ void __launch_bounds__(256) vtw_flat_kernel(const T* __restrict__ V, int64_t N, int rt, int P,
                                                       const T* __restrict__ w, T* __restrict__ partial) {
  constexpr int UNR = 4;
  __shared__ T red[256 * VW];
  const int nt = P * rt / VW;
  const int64_t groups = (N + P - 1) / P;
  const int64_t per = (groups + gridDim.x - 1) / gridDim.x;
  const int64_t g0 = (int64_t)blockIdx.x * per, g1 = std::min<int64_t>(groups, g0 + per);
  for (int tb = 0; tb < nt; tb += 256) {  // more than 256 units a group: one pass per 256
    const int width = std::min(256, nt - tb), lanes = 256 / width;
    const int t = tb + threadIdx.x % width, gl = threadIdx.x / width;
    const bool on = gl < lanes;
    int off[VW];
    T acc[UNR][VW];
#pragma unroll
    for (int e = 0; e < VW; ++e) {
      off[e] = (VW * t + e) / rt;
#pragma unroll
      for (int u = 0; u < UNR; ++u) acc[u][e] = T(0);
    }
    auto load = [&](int64_t g, T* v) {
      const T* src = V + g * P * rt + (int64_t)VW * t;
      if constexpr (VW == 4) {
        const float4 x = *reinterpret_cast<const float4*>(src);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
      } else if constexpr (VW == 2) {
        const double2 x = *reinterpret_cast<const double2*>(src);
        v[0] = x.x; v[1] = x.y;
      } else {
        v[0] = *src;
      }
    };
    if (on) {
      // groups that lie wholly inside N; the last one may not
      const int64_t gfull = std::min<int64_t>(g1, N / P);
      int64_t g = g0 + gl;
      for (; g + (UNR - 1) * lanes < gfull; g += UNR * lanes) {
        T v[UNR][VW];
#pragma unroll
        for (int u = 0; u < UNR; ++u) load(g + u * lanes, v[u]);
#pragma unroll
        for (int u = 0; u < UNR; ++u)
#pragma unroll
          for (int e = 0; e < VW; ++e) acc[u][e] = fma(v[u][e], w[(g + u * lanes) * P + off[e]], acc[u][e]);
      }
      for (; g < gfull; g += lanes) {
        T v[VW];
        load(g, v);
#pragma unroll
        for (int e = 0; e < VW; ++e) acc[0][e] = fma(v[e], w[g * P + off[e]], acc[0][e]);
      }
      if (g < g1)
#pragma unroll
        for (int e = 0; e < VW; ++e) {
          const int64_t row = g * P + off[e];
          if (row < N) acc[0][e] = fma(V[g * P * rt + (int64_t)VW * t + e], w[row], acc[0][e]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < VW; ++e) red[threadIdx.x * VW + e] = (acc[0][e] + acc[1][e]) + (acc[2][e] + acc[3][e]);
    __syncthreads();
    // the lanes' sums, halved until few are left (few columns have up to 256 lanes)
    int left = lanes;
    while (left > 16) {
      const int half = (left + 1) / 2;
      if (gl + half < left)
#pragma unroll
        for (int e = 0; e < VW; ++e) red[threadIdx.x * VW + e] += red[(threadIdx.x + half * width) * VW + e];
      left = half;
      __syncthreads();
    }
    // element VW t + e of a group is column (VW t + e) mod rt; red holds elements VW tb ..
    for (int c = threadIdx.x; c < rt; c += 256) {
      T sum = T(0);
      for (int el = c; el < P * rt; el += rt) {
        const int q = el - VW * tb;
        if (q < 0 || q >= VW * width) continue;
        for (int l = 0; l < left; ++l) sum += red[l * width * VW + q];
      }
      T* dst = partial + (int64_t)blockIdx.x * rt + c;
      *dst = tb == 0 ? sum : *dst + sum;
    }
    __syncthreads();
  }
}

// The form of V^T w: the flat one (true; *P rows a unit group, *VW elements a unit) or the columns. What bounds both is the
// read of V. By single elements, for a V that is not 16-byte aligned, the flat form is the better one up to 32 columns, where
// the column form leaves half of its 64 column threads idle (100k x 12 FP64: 62 us against 70, the whole product), and far worse
// beyond (100k x 129 FP32: 47 us against 14). By 16-byte units, where its units occupy enough of the block's threads,
//  - FP32 takes it (with the read of U after it, 100k x 177: 49 us against 55; 400k x 257: 172 against 226). Odd ranks from
//    129 to 153, whose units of four rows leave 40 % of the threads idle, stay with the columns (100k x 129: 39
//    against 35) unless V is too large for L2 (400k x 129: 118 against 137);
//  - FP64, whose units hold two columns, gains up to 32 columns (400k x 12: 178 us against 211) and where V does not stay in
//    L2 (400k x 257: 527 against 582); in between the columns are the faster ones (100k x 63: 76 against 80, 50k x 177: 88
//    against 111).
template <typename T>
bool vtw_flat(const T* V, int64_t N, int rt, int* P, int* VW) {
  *P = *VW = 1;
  if ((reinterpret_cast<uintptr_t>(V) & 15) != 0) return rt <= 32;
  constexpr int W = 16 / (int)sizeof(T);
  *VW = W;
  *P = rt % W == 0 ? 1 : W % 2 == 0 && (2 * rt) % W == 0 ? 2 : W;
  const int nt = *P * rt / W, busy = nt >= 256 ? 256 : 256 / nt * nt;  // threads at work
  const bool large = (double)N * rt * sizeof(T) > 129e6;
  if (sizeof(T) == 4) return busy >= 154 || rt > 256 || large;
  return rt <= 32 || (rt > 64 && busy >= 218 && large);
}

// t = sum over the partial rows, written into row 0 of `partial`: 32 columns x 8 part lanes
// per block, each lane summing every eighth part, the lanes then added in a fixed order (the
// rows a block reads belong to its own columns only).
template <typename T>
__global__ void __launch_bounds__(256) reduce_parts_kernel(T* __restrict__ partial, int nparts, int rt) {
  __shared__ T red[8][32];
  const int cl = threadIdx.x & 31, pl = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * 32 + cl;
  T acc = T(0);
  if (c < rt)
    for (int b = pl; b < nparts; b += 8) acc += partial[(int64_t)b * rt + c];
  red[pl][cl] = acc;
  __syncthreads();
  if (pl == 0 && c < rt)
    partial[c] = ((red[0][cl] + red[1][cl]) + (red[2][cl] + red[3][cl])) +
                 ((red[4][cl] + red[5][cl]) + (red[6][cl] + red[7][cl]));
}

// s = M t, one warp per row of M (rs x rt, row-major); t is the sum of the nparts rows of `partial` (one row
// once reduce_parts_kernel has run; a few where the sum is cheaper than that launch), formed by
// each block in shared memory 1024 columns at a time.
template <typename T>
__global__ void __launch_bounds__(256) mt_kernel(const T* __restrict__ M, int rs, int rt,
                                                 const T* __restrict__ partial, int nparts, T* __restrict__ s_out) {
  __shared__ T t[1024];
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  T acc = T(0);
  for (int c0 = 0; c0 < rt; c0 += 1024) {
    const int w = std::min(1024, rt - c0);
    __syncthreads();
    for (int c = threadIdx.x; c < w; c += 256) {
      T sum = T(0);
      for (int b = 0; b < nparts; ++b) sum += partial[(int64_t)b * rt + c0 + c];
      t[c] = sum;
    }
    __syncthreads();
    if (r < rs) {
      const T* m = M + r * rt + c0;
      for (int c = lane; c < w; c += 32) acc = fma(m[c], t[c], acc);
    }
  }
  acc = warp_sum<T>(acc);
  if (lane == 0 && r < rs) s_out[r] = acc;
}

// out[p] = U[p, :] . s, a warp taking R consecutive rows at a time (their loads are all in
// flight before any is reduced); s is read through the L1 cache. What bounds it: the read of U. Four rows up to 128
// columns, two beyond, on more blocks (four: 1M x 45 FP32 127 -> 140 us with two, the read of V before it included; two:
// 50k x 516 FP32 143 -> 134, 5,000 x 180 FP64 31 -> 29).
template <typename T, int R>
__global__ void __launch_bounds__(256) us_kernel(const T* __restrict__ U, int64_t N, int rs,
                                                 const T* __restrict__ s, T* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t row = R * (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5); row < N; row += R * nw) {
    const int live = (int)std::min<int64_t>(R, N - row);
    const T* u = U + row * rs;
    T acc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = T(0);
    if (live == R) {
#pragma unroll 4
      for (int c = lane; c < rs; c += 32) {
        const T sc = __ldg(s + c);
#pragma unroll
        for (int i = 0; i < R; ++i) acc[i] = fma(u[(int64_t)i * rs + c], sc, acc[i]);
      }
    } else {
      for (int c = lane; c < rs; c += 32) {
        const T sc = __ldg(s + c);
#pragma unroll
        for (int i = 0; i < R; ++i)
          if (i < live) acc[i] = fma(u[(int64_t)i * rs + c], sc, acc[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = warp_sum<T>(acc[i]);
#pragma unroll
    for (int i = 0; i < R; ++i)
      if (lane == i && i < live) out[row + i] = acc[i];
  }
}

template <typename T>
pttk_status apply_typed(const T* U, const T* M, const T* V, int64_t N_s, int64_t N_t, int rs,
                        int rt, const T* w, T* out, T* scratch, int nparts, cudaStream_t s) {
  T* partial = scratch;
  T* sv = scratch + (size_t)nparts * rt;
  PTTK_PROF("apply", s);
  if (N_t > 0) {
    int P, VW;
    if (!vtw_flat(V, N_t, rt, &P, &VW)) vtw_columns_kernel<T><<<nparts, 256, 0, s>>>(V, N_t, rt, w, partial);
    else if (VW == 1) vtw_flat_kernel<T, 1><<<nparts, 256, 0, s>>>(V, N_t, rt, P, w, partial);
    else vtw_flat_kernel<T, 16 / (int)sizeof(T)><<<nparts, 256, 0, s>>>(V, N_t, rt, P, w, partial);
    pttk::count_launch();
  } else {
    PTTK_CUDA(cudaMemsetAsync(partial, 0, sizeof(T) * (size_t)nparts * rt, s));
  }
  int left = nparts;
  if (nparts > 32) {
    reduce_parts_kernel<T><<<(unsigned)((rt + 31) / 32), 256, 0, s>>>(partial, nparts, rt); pttk::count_launch();
    left = 1;
  }
  mt_kernel<T><<<(unsigned)((rs + 7) / 8), 256, 0, s>>>(M, rs, rt, partial, left, sv); pttk::count_launch();
  if (N_s > 0) {
    const int R = rs <= 128 ? 4 : 2;
    const unsigned blocks = (unsigned)std::min<int64_t>((N_s * (32 / R) + 255) / 256, (int64_t)sm_count() * (32 / R));
    if (R == 4) us_kernel<T, 4><<<blocks, 256, 0, s>>>(U, N_s, rs, sv, out);
    else us_kernel<T, 2><<<blocks, 256, 0, s>>>(U, N_s, rs, sv, out);
    pttk::count_launch();
  }
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

int apply_parts(int64_t N_t) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((N_t + 255) / 256, (int64_t)sm_count() * 4));
}

}  // namespace

// ---------------- point domain ---------------------------------------------------------
// The problem is stated for X in B_s and Y in B_t (Section 1). One pass over a point set
// records PTTK_EDOMAIN in the handle's status word if any coordinate lies outside its
// interval by more than a relative slack of 1e-12. FP32 points are compared with the
// FP32-rounded interval ends: rounding is monotone, so a point inside the box stays inside
// the rounded box when it is cast. Both sides are checked in one launch (blockIdx.y picks
// the side). The pass is a plain read of the point sets (12 B per point for d = 3 in FP32),
// so nothing in it may use the FP64 pipe, which runs at about 2 operations per clock per SM:
//  - FP32 points are compared in FP32 with bounds rounded inwards on the host (the smallest
//    float >= lo - slack, the largest float <= hi + slack), which accepts exactly the floats
//    the FP64 comparison accepts;
//  - FP64 points are compared as order-preserving 64-bit integer keys of their bit patterns.
// A NaN coordinate fails both forms of the comparison. A side whose base is 16-byte aligned
// and whose N d elements fill whole 16-byte units is read with 16-byte loads, else element by
// element. The coordinate index is carried from step to step instead of taken modulo d, and
// the bounds sit in shared memory.
struct PointCheck {
  const void* P[2];
  int64_t total[2];                        // N * d elements per side
  int vec[2];                              // 16-byte loads: base 16-byte aligned, total a multiple of 16 B
  long long klo[2][PTTK_MAX_D], khi[2][PTTK_MAX_D];  // FP64 points: integer keys of the bounds
  float flo[2][PTTK_MAX_D], fhi[2][PTTK_MAX_D];      // FP32 points: the bounds as floats
};

// Key of a double: a signed 64-bit integer ordered as the doubles are, with -0 and +0 equal
// (the magnitude bits, negated for a set sign bit). A NaN's key lies beyond the keys of the
// infinities on its sign's side, so it fails any comparison with finite bounds.
__host__ __device__ __forceinline__ long long order_key(long long bits) {
  return bits < 0 ? -(bits & 0x7FFFFFFFFFFFFFFFLL) : bits;
}

template <typename T>
__global__ void __launch_bounds__(256) point_domain_kernel(PointCheck a, int d, int* __restrict__ status) {
  constexpr bool F64 = std::is_same_v<T, double>;
  using B = std::conditional_t<F64, long long, float>;
  constexpr int W = 16 / (int)sizeof(T);  // elements per 16-byte load
  __shared__ B lo[PTTK_MAX_D], hi[PTTK_MAX_D];
  const int side = blockIdx.y;
  if (threadIdx.x < d) {
    if constexpr (F64) {
      lo[threadIdx.x] = a.klo[side][threadIdx.x];
      hi[threadIdx.x] = a.khi[side][threadIdx.x];
    } else {
      lo[threadIdx.x] = a.flo[side][threadIdx.x];
      hi[threadIdx.x] = a.fhi[side][threadIdx.x];
    }
  }
  __syncthreads();
  bool bad = false;
  auto check = [&](B x, int c) {
    if constexpr (F64) bad |= order_key(x) < lo[c] || order_key(x) > hi[c];
    else bad |= !(x >= lo[c] && x <= hi[c]);  // also catches NaN
  };
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a.vec[side]) {
    // e counts 16-byte units; the coordinate of the unit's first element is carried
    const int64_t units = a.total[side] / W;
    int c = (int)((e * W) % d);
    const int cstep = (int)((stride * W) % d);
    using V = std::conditional_t<F64, longlong2, float4>;
    const V* __restrict__ P = static_cast<const V*>(a.P[side]);
#pragma unroll 2
    for (; e < units; e += stride) {
      const V v = __ldg(P + e);
      int cc = c;
      if constexpr (F64) {
        check(v.x, cc);
        cc = cc + 1 == d ? 0 : cc + 1;
        check(v.y, cc);
      } else {
        check(v.x, cc);
        cc = cc + 1 == d ? 0 : cc + 1;
        check(v.y, cc);
        cc = cc + 1 == d ? 0 : cc + 1;
        check(v.z, cc);
        cc = cc + 1 == d ? 0 : cc + 1;
        check(v.w, cc);
      }
      c += cstep;
      if (c >= d) c -= d;
    }
  } else {
    const int64_t total = a.total[side];
    int c = (int)(e % d);
    const int cstep = (int)(stride % d);
    const B* __restrict__ P = static_cast<const B*>(a.P[side]);
#pragma unroll 4
    for (; e < total; e += stride) {
      check(__ldg(P + e), c);
      c += cstep;
      if (c >= d) c -= d;
    }
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicCAS(status, 0, (int)PTTK_EDOMAIN);
}

// The smallest float >= v and the largest float <= v.
static float float_at_or_above(double v) {
  float f = (float)v;
  if ((double)f < v) f = std::nextafter(f, std::numeric_limits<float>::infinity());
  return f;
}
static float float_at_or_below(double v) {
  float f = (float)v;
  if ((double)f > v) f = std::nextafter(f, -std::numeric_limits<float>::infinity());
  return f;
}
static long long key_of(double v) {
  long long bits;
  std::memcpy(&bits, &v, sizeof bits);
  return order_key(bits);
}

pttk_status point_domain_check(const pttk_tt* tt, const void* X, int64_t N_s, const void* Y, int64_t N_t, bool fp64,
                               int* status, cudaStream_t s) {
  N_s = X ? std::max<int64_t>(N_s, 0) : 0;
  N_t = Y ? std::max<int64_t>(N_t, 0) : 0;
  if (N_s == 0 && N_t == 0) return PTTK_OK;
  PTTK_PROF("domain", s);
  PointCheck a{};
  a.P[0] = X;
  a.P[1] = Y;
  a.total[0] = N_s * tt->d;
  a.total[1] = N_t * tt->d;
  for (int side = 0; side < 2; ++side)
    for (int c = 0; c < tt->d; ++c) {
      const int bj = side == 0 ? c : tt->d + tt->dtheta + c;
      const double lo = tt->box[bj][0], hi = tt->box[bj][1], slack = 1e-12 * (hi - lo);
      a.klo[side][c] = key_of(lo - slack);
      a.khi[side][c] = key_of(hi + slack);
      a.flo[side][c] = float_at_or_above((double)(float)lo - slack);
      a.fhi[side][c] = float_at_or_below((double)(float)hi + slack);
    }
  const int W = fp64 ? 2 : 4;
  int64_t work = 0;
  for (int side = 0; side < 2; ++side) {
    a.vec[side] = (reinterpret_cast<uintptr_t>(a.P[side]) & 15) == 0 && a.total[side] % W == 0;
    work = std::max(work, a.vec[side] ? a.total[side] / W : a.total[side]);
  }
  const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, (int64_t)sm_count() * 4)), 2);
  if (fp64) point_domain_kernel<double><<<grid, 256, 0, s>>>(a, tt->d, status);
  else point_domain_kernel<float><<<grid, 256, 0, s>>>(a, tt->d, status);
  pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

// Step `step` of a side's chain: dimensions of its oriented core and the point coordinate.
int oriented_core_dims(const pttk_tt* tt, bool source, int step, int* R_in, int* R_out,
                       int* coord) {
  if (source) {
    const int k = step;  // core G_{k+1}
    *R_in = tt->ranks[k];
    *R_out = tt->ranks[k + 1];
    *coord = step;
    return k;
  }
  const int k = tt->D - 1 - step;  // core G_{D-step}, read transposed
  *R_in = tt->ranks[k + 1];
  *R_out = tt->ranks[k];
  *coord = tt->d - 1 - step;
  return k;
}

pttk_status theta_core_run(const pttk_tt* tt, const double* theta_hat, bool fp64, void* M,
                           cudaStream_t s) {
  const int d = tt->d, dth = tt->dtheta, n = tt->n;
  const int rs = tt->ranks[d], rt = tt->ranks[d + dth];
  if (dth == 0) {
    identity_rowmajor_kernel<<<64, 256, 0, s>>>(M, rs, fp64); pttk::count_launch();
    PTTK_CUDA(cudaGetLastError());
    return PTTK_OK;
  }
  PTTK_PROF("theta_core", s);
  ThetaCores c{};
  int64_t most = 0;
  for (int j = 0; j < dth; ++j) {
    c.G[j] = tt->cores64 + tt->core_off[d + j];
    c.th[j] = theta_hat[j];
    c.ra[j] = tt->ranks[d + j];
    c.rb[j] = tt->ranks[d + j + 1];
    most = std::max(most, (int64_t)c.ra[j] * c.rb[j]);
  }
  const dim3 cgrid((unsigned)std::min<int64_t>((most + 255) / 256, sm_count() * 8), (unsigned)dth);
  if (dth == 1) {
    if (fp64) contract_theta_kernel<double><<<cgrid, 256, 0, s>>>(c, n, static_cast<double*>(M));
    else contract_theta_kernel<float><<<cgrid, 256, 0, s>>>(c, n, static_cast<float*>(M));
    pttk::count_launch();
    PTTK_CUDA(cudaGetLastError());
    return PTTK_OK;
  }
  const int rm = tt->ranks[d + 1];
  const int nslices = (rm + HP_T - 1) / HP_T;
  const size_t e1 = (size_t)rs * rm, e2 = (size_t)rm * rt;
  double* work = nullptr;
  PTTK_CUDA(ws_malloc(&work, sizeof(double) * (e1 + e2 + (size_t)rs * rt * nslices), s));
  c.out[0] = work;
  c.out[1] = work + e1;
  double* part = work + e1 + e2;
  contract_theta_kernel<double><<<cgrid, 256, 0, s>>>(c, n, nullptr); pttk::count_launch();
  const unsigned blocks = (unsigned)std::min<int64_t>(((int64_t)rs * rt + 255) / 256, sm_count() * 8);
  const dim3 grid((unsigned)((rs + HP_T - 1) / HP_T), (unsigned)((rt + HP_T - 1) / HP_T), (unsigned)nslices);
  hprod_splitk_kernel<<<grid, 256, 0, s>>>(c.out[0], c.out[1], rs, rm, rt, part); pttk::count_launch();
  if (fp64) { hprod_reduce_kernel<double><<<blocks, 256, 0, s>>>(part, nslices, rs, rt, static_cast<double*>(M)); pttk::count_launch(); }
  else { hprod_reduce_kernel<float><<<blocks, 256, 0, s>>>(part, nslices, rs, rt, static_cast<float*>(M)); pttk::count_launch(); }
  const cudaError_t err = cudaGetLastError();
  cudaFreeAsync(work, s);
  PTTK_CUDA(err);
  return PTTK_OK;
}

// Oriented core pointer for a chain step (see pttk_tt::oriented).
const void* oriented_core_ptr(const pttk_tt* tt, bool source, int k, bool fp64);

template <typename T, int TM>
static pttk_status launch_chain(ChainArgs a, int ct_max, cudaStream_t s) {
  constexpr int P = 16 * TM;
  const size_t smem = sizeof(T) * ((size_t)2 * P * a.rin_max + (size_t)P * a.n + 2 * BK * P + 2 * BK * (ct_max + 2));
  auto kfn = ct_max <= 64 ? chain_kernel<T, TM, 64> : chain_kernel<T, TM, sizeof(T) == 8 ? 96 : 128>;
  PTTK_CUDA(allow_smem((const void*)kfn));
  a.blocks0 = (a.side[0].N + P - 1) / P;
  const int64_t blocks = a.blocks0 + (a.side[1].N + P - 1) / P;
  PTTK_PROF("chain", s);
  kfn<<<(unsigned)blocks, 256, smem, s>>>(a); pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

// Both sides' factors (a side with N = 0 is left out) in one launch.
static pttk_status chain_run(const pttk_tt* tt, const void* X, int64_t N_s, const void* Y, int64_t N_t, pttk_prec prec,
                             void* U, void* V, cudaStream_t s, int nsteps) {
  if (N_s == 0 && N_t == 0) return PTTK_OK;
  const bool fp64 = prec == PTTK_FP64;
  ChainArgs a{};
  a.nsteps = (nsteps > 0 && nsteps < tt->d) ? nsteps : tt->d;
  a.n = tt->n;
  a.d = tt->d;
  a.rin_max = 1;
  int rmax = 1, ct_max = 0;
  for (int sd = 0; sd < 2; ++sd) {
    ChainSide& side = a.side[sd];
    side.pts = sd == 0 ? X : Y;
    side.out = sd == 0 ? U : V;
    side.N = sd == 0 ? N_s : N_t;
    if (side.N == 0) continue;
    for (int i = 0; i < a.nsteps; ++i) {
      int rin, rout, coord;
      const int k = oriented_core_dims(tt, sd == 0, i, &rin, &rout, &coord);
      ChainStep& st = side.st[i];
      st.G = oriented_core_ptr(tt, sd == 0, k, fp64);
      st.R_in = rin;
      st.R_out = rout;
      st.coord = coord;
      st.magic = (uint32_t)((0x100000000ull + rin - 1) / rin);
      // The pass width with the fewest padded columns, the widest of equals; FP64 takes no 128, whose
      // accumulators would leave room for one block an SM.
      st.ct = 0;
      if (rout > NARROW) {
        st.ct = 64;
        for (int ct : {96, 128})
          if ((ct == 96 || !fp64) && (rout + ct - 1) / ct * ct <= (rout + st.ct - 1) / st.ct * st.ct) st.ct = ct;
      }
      ct_max = std::max(ct_max, st.ct);
      const int bj = sd == 0 ? coord : tt->d + tt->dtheta + coord;
      st.lo = tt->box[bj][0];
      st.hi = tt->box[bj][1];
      a.rin_max = std::max(a.rin_max, rin);
      rmax = std::max(rmax, std::max(rin, rout));
    }
  }
  // the ranks taken: 16 points' rows of the widest rank, padded to 64, twice within 200,000 bytes
  const size_t elem = fp64 ? 8 : 4;
  const size_t budget = 200000;
  const size_t rpad = (size_t)(rmax + 63) / 64 * 64;
  if (elem * (2 * 16 * rpad + 16 * PTTK_MAX_N + 16 * 16 + 16 * 64) > budget)
    return set_error(PTTK_ENOTSUP, "TT ranks too large for the SIMT factor chain");
  // The most points per block that shared memory holds and that still give every SM a block (a block's
  // time hardly falls with its points, so few points want more blocks): FP32 up to 128, FP64 up to 64.
  int tm = fp64 ? 4 : 8;
  auto smem_of = [&](int t) {
    const size_t P = 16 * (size_t)t;
    return elem * (2 * P * a.rin_max + P * a.n + 2 * BK * P + 2 * BK * ((size_t)ct_max + 2));
  };
  auto blocks_of = [&](int t) { return (N_s + 16 * t - 1) / (16 * t) + (N_t + 16 * t - 1) / (16 * t); };
  while (tm > 1 && (smem_of(tm) > 227 * 1024 || blocks_of(tm) < sm_count())) tm /= 2;
  if (smem_of(tm) > 227 * 1024) return set_error(PTTK_ENOTSUP, "TT ranks too large for the SIMT factor chain");
  if (fp64) {
    if (tm == 4) return launch_chain<double, 4>(a, ct_max, s);
    if (tm == 2) return launch_chain<double, 2>(a, ct_max, s);
    return launch_chain<double, 1>(a, ct_max, s);
  }
  if (tm == 8) return launch_chain<float, 8>(a, ct_max, s);
  if (tm == 4) return launch_chain<float, 4>(a, ct_max, s);
  if (tm == 2) return launch_chain<float, 2>(a, ct_max, s);
  return launch_chain<float, 1>(a, ct_max, s);
}

pttk_status factor_build_run(const pttk_tt* tt, bool source, const void* P, int64_t N, pttk_prec prec, void* out,
                             cudaStream_t s, int nsteps) {
  return source ? chain_run(tt, P, N, nullptr, 0, prec, out, nullptr, s, nsteps)
                : chain_run(tt, nullptr, 0, P, N, prec, nullptr, out, s, nsteps);
}

pttk_status factor_build_both(const pttk_tt* tt, const void* X, int64_t N_s, const void* Y, int64_t N_t, pttk_prec prec,
                              void* U, void* V, cudaStream_t s) {
  return chain_run(tt, X, N_s, Y, N_t, prec, U, V, s, 0);
}

size_t apply_scratch_bytes(int64_t N_t, int rs, int rt, bool fp64) {
  const int nparts = apply_parts(N_t);
  return (fp64 ? 8 : 4) * ((size_t)nparts * rt + (size_t)rs);
}

pttk_status apply_run(const void* U, const void* M, const void* V, int64_t N_s, int64_t N_t,
                      int rs, int rt, bool fp64, const void* w, void* out, void* scratch,
                      cudaStream_t s) {
  const int nparts = apply_parts(N_t);
  if (fp64)
    return apply_typed<double>(static_cast<const double*>(U), static_cast<const double*>(M),
                               static_cast<const double*>(V), N_s, N_t, rs, rt,
                               static_cast<const double*>(w), static_cast<double*>(out),
                               static_cast<double*>(scratch), nparts, s);
  return apply_typed<float>(static_cast<const float*>(U), static_cast<const float*>(M),
                            static_cast<const float*>(V), N_s, N_t, rs, rt,
                            static_cast<const float*>(w), static_cast<float*>(out),
                            static_cast<float*>(scratch), nparts, s);
}

}  // namespace pttk

// ---------------- apply without device allocation ---------------------------------------
// pttk_apply_noalloc runs the same kernels as pttk_apply, with its scratch (the per-block
// partial sums of V^T w and the vector M (V^T w)) in this file-scope device array instead of
// a stream-ordered allocation. Every device that loads the library holds the array until the
// process exits. All calls share it, so calls whose work overlaps on the GPU race.
namespace pttk {
namespace {

constexpr size_t kNoAllocScratchBytes = 1u << 20;  // 1 MiB
static __device__ __align__(256) unsigned char g_apply_scratch[kNoAllocScratchBytes];

std::mutex g_scratch_mu;
void* g_scratch_dev[64] = {nullptr};

// Device address of g_apply_scratch on the current device, looked up once per device.
// In host code the symbol name is only a host-side stand-in, never a device address.
pttk_status scratch_address(void** out) {
  int dev = 0;
  PTTK_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return set_error(PTTK_EINVAL, "device ordinal above 63");
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_dev[dev]) {
    void* p = nullptr;
    PTTK_CUDA(cudaGetSymbolAddress(&p, g_apply_scratch));
    g_scratch_dev[dev] = p;
  }
  *out = g_scratch_dev[dev];
  return PTTK_OK;
}

}  // namespace
}  // namespace pttk

extern "C" pttk_status pttk_apply_noalloc(const void* U, const void* M, const void* V, int64_t N_s,
                                          int64_t N_t, int rs, int rt, pttk_prec prec, const void* w,
                                          void* out, void* stream) {
  using namespace pttk;
  clear_error();
  if (!M || (N_s > 0 && (!U || !out)) || (N_t > 0 && (!V || !w))) return set_error(PTTK_EINVAL, "NULL argument");
  if (N_s < 0 || N_t < 0 || rs < 1 || rt < 1) return set_error(PTTK_EINVAL, "bad size");
  if (prec != PTTK_FP64 && prec != PTTK_FP32) return set_error(PTTK_EINVAL, "apply precision must be FP64 or FP32");
  const bool fp64 = prec == PTTK_FP64;
  const size_t elem = fp64 ? 8 : 4;
  const size_t cap = kNoAllocScratchBytes / elem;
  if ((size_t)rs + (size_t)rt > cap) {
    char buf[200];
    snprintf(buf, sizeof buf,
             "pttk_apply_noalloc: rs + rt = %lld exceeds its fixed scratch of %zu %s elements",
             (long long)rs + rt, cap, fp64 ? "FP64" : "FP32");
    return set_error(PTTK_EINVAL, buf);
  }
  void* scratch = nullptr;
  PTTK_TRY(scratch_address(&scratch));
  // as many partial-sum blocks as pttk_apply uses, fewer if they would not fit
  const int nparts = (int)std::max<int64_t>(
      1, std::min<int64_t>(apply_parts(N_t), (int64_t)((cap - (size_t)rs) / (size_t)rt)));
  cudaStream_t s = as_stream(stream);
  if (fp64)
    return apply_typed<double>(static_cast<const double*>(U), static_cast<const double*>(M),
                               static_cast<const double*>(V), N_s, N_t, rs, rt,
                               static_cast<const double*>(w), static_cast<double*>(out),
                               static_cast<double*>(scratch), nparts, s);
  return apply_typed<float>(static_cast<const float*>(U), static_cast<const float*>(M),
                            static_cast<const float*>(V), N_s, N_t, rs, rt,
                            static_cast<const float*>(w), static_cast<float*>(out),
                            static_cast<float*>(scratch), nparts, s);
}
