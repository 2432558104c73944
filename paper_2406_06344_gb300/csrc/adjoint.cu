// Adjoint of the scalar loss L = w^T K~ z = w^T U(X) H(theta) V(Y)^T z.
//
// With a = U^T w, b = V^T z and g = H b:
//   L = a . g;
//   dL/dtheta_j = a^T H_1 ... H_j' ... H_dtheta b,  H_j' = sum_k G_{d+j}[:, k, :] T_k'(thetahat_j)
//                 dthetahat_j/dtheta_j (Eq. hmat differentiated; dthetahat/dtheta = 2/(lo - hi)
//                 for the printed interval map);
//   dL/dX: reverse pass through the chain of Algorithm 2, Phase 3 for every source point. The
//   adjoint of the chain output for point p is w_p g (rank one over the points), so the last
//   step needs only the vector q = G_d^{2} g; earlier steps take Q_i = gbar_i G_i^{2 T}. Step i
//   (S_out = (B_i face-split S_in) G_i^{2}) propagates
//     dB_i[p, j]   = sum_a S_in[p, a] Q_i[p, a + R_in j],
//     gbar_in[p,a] = sum_j B_i[p, j] Q_i[p, a + R_in j],
//     dL/dx_{p,i}  = sum_j dB_i[p, j] T_j'(xhat_{p,i}) 2/(lo_i - hi_i).
//   The Chebyshev bases and their derivatives (T_0' = 0, T_1' = 1,
//   T_{j+1}' = 2 T_j + 2 x T_j' - T_{j-1}') are recomputed per point, never stored; the chain
//   intermediates S_1..S_{d-1} come from rerunning the (cheap) leading steps of the chain.
#include <math.h>

#include <algorithm>
#include <vector>

#include "pttk_internal.cuh"

namespace pttk {
pttk_status factor_build_tc(const pttk_tt* tt, TcImageCache* cache, const float* X, int64_t N_s,
                            const float* Y, int64_t N_t, pttk_prec prec, float* U, float* V,
                            int* d_status, int cfg, cudaStream_t s);
namespace {

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// A float as a double. The conversion instruction takes the FP64 pipe twice as long as an FMA here; for a
// normal number the same bits come from four integer operations (the rare branch is volatile so that
// the conversion is not computed ahead of it).
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x), e = b & 0x7f800000u;
  if (e == 0 || e == 0x7f800000u) {
    double d;
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(x));
    return d;
  }
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }
// The same for K values with one branch for all of them.
template <int K>
__device__ __forceinline__ void widen_all(const float (&x)[K], double (&y)[K]) {
  bool rare = false;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int b = __float_as_int(x[k]);
    rare |= (uint32_t)(b & 0x7f800000) - 0x00800000u >= 0x7f000000u;
    y[k] = __hiloint2double(((b >> 3) & (int)0x8fffffff) + 0x38000000, b << 29);
  }
  if (rare)
#pragma unroll
    for (int k = 0; k < K; ++k) y[k] = widen(x[k]);
}
template <int K>
__device__ __forceinline__ void widen_all(const double (&x)[K], double (&y)[K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) y[k] = x[k];
}

// partial[(4 blk + lane) r + c] = sum over every fourth of the block's rows of A[row, c] w[row] in FP64
// (A: N x r row-major). Threads are 4 row lanes x 64 column groups of VW consecutive columns (VW = 4
// when the rows are 16-byte aligned, else 1), four or eight rows of loads in flight each, whose rare values share
// one branch. What bounds it: the FP64 pipe (500k x 177: 0.145 ms) and the widening; 0.56 -> 0.22 ms.
template <typename T, int VW>
__global__ void __launch_bounds__(256) weighted_colsum(const T* __restrict__ A, const T* __restrict__ w,
                                                       int64_t N, int r, double* __restrict__ partial) {
  const int64_t per = (N + gridDim.x - 1) / gridDim.x;
  const int64_t r0 = (int64_t)blockIdx.x * per, r1 = std::min<int64_t>(N, r0 + per);
  const int cl = threadIdx.x & 63, rl = threadIdx.x >> 6;
  for (int c = cl * VW; c < r; c += 64 * VW) {  // with VW = 4, r is a multiple of 4
    double acc[VW];
#pragma unroll
    for (int q = 0; q < VW; ++q) acc[q] = 0.0;
    int64_t i = r0 + rl;
    constexpr int R = VW == 1 ? 8 : 4;  // rows in flight
    for (; i + 4 * (R - 1) < r1; i += 4 * R) {
      T v[R * VW], wr[R];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const T* src = A + (i + 4 * u) * r + c;
        wr[u] = w[i + 4 * u];
        if constexpr (VW == 4 && sizeof(T) == 4) {
          const float4 x = *reinterpret_cast<const float4*>(src);
          v[4 * u] = x.x; v[4 * u + 1] = x.y; v[4 * u + 2] = x.z; v[4 * u + 3] = x.w;
        } else {
#pragma unroll
          for (int q = 0; q < VW; ++q) v[VW * u + q] = src[q];
        }
      }
      double vd[R * VW], wd[R];
      widen_all(v, vd);
      widen_all(wr, wd);
#pragma unroll
      for (int u = 0; u < R; ++u)
#pragma unroll
        for (int q = 0; q < VW; ++q) acc[q] = fma(vd[VW * u + q], wd[u], acc[q]);
    }
    for (; i < r1; i += 4) {
      const double wr = widen(w[i]);
#pragma unroll
      for (int q = 0; q < VW; ++q) acc[q] = fma(widen(A[i * r + c + q]), wr, acc[q]);
    }
#pragma unroll
    for (int q = 0; q < VW; ++q) partial[(4 * (int64_t)blockIdx.x + rl) * r + c + q] = acc[q];
  }
}

// out[c] = sum over the partial rows, one block per column, in a fixed order
__global__ void __launch_bounds__(256) sum_partials(const double* __restrict__ partial, int nparts, int r,
                                                    double* __restrict__ out) {
  __shared__ double red[8];
  const int c = blockIdx.x;
  double acc = 0.0;
  for (int b = threadIdx.x; b < nparts; b += 256) acc += partial[(int64_t)b * r + c];
  acc = warp_sum_d(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) acc += red[k];
    out[c] = acc;
  }
}

// Chebyshev values T_k(x) (deriv = 0) or T_k'(x) * scale (deriv = 1), k < n, into t[0..n)
__device__ void cheb_row(double x, int n, bool deriv, double scale, double* t) {
  double t0 = 1.0, t1 = x, d0 = 0.0, d1 = 1.0;
  for (int k = 0; k < n; ++k) {
    if (k == 0) t[k] = deriv ? 0.0 : 1.0;
    else if (k == 1) t[k] = deriv ? scale : x;
    else {
      const double t2 = 2.0 * x * t1 - t0;
      const double d2 = 2.0 * t1 + 2.0 * x * d1 - d0;
      t[k] = deriv ? d2 * scale : t2;
      t0 = t1;
      t1 = t2;
      d0 = d1;
      d1 = d2;
    }
  }
}

// Contractions of theta cores G (ra x n x rb, column-major) with the Chebyshev (or derivative) vector of
// th, applied to a vector on one side, up to four in one launch (blockIdx.y), one block per output:
//   left  (side 0): out[c] = sum_{a,k} x[a] G[a, k, c] t[k]      (x: ra, out: rb)
//   right (side 1): out[a] = sum_{k,c} G[a, k, c] t[k] x[c]      (x: rb, out: ra)
// A block's 256 threads keep their loads in flight together: what bounds it is their latency.
struct CoreVec {
  const double* G;
  const double* x;
  double* out;
  double th, scale;
  int ra, rb, side, deriv;
};
struct CoreVecs {
  CoreVec t[4];
};
__global__ void __launch_bounds__(256) core_vecs(CoreVecs v, int n) {
  const CoreVec c = v.t[blockIdx.y];
  const int o = blockIdx.x;
  if (o >= (c.side == 0 ? c.rb : c.ra)) return;
  __shared__ double t[PTTK_MAX_N];
  __shared__ double red[8];
  if (threadIdx.x == 0) {
    double tl[PTTK_MAX_N];
    cheb_row(c.th, n, c.deriv != 0, c.scale, tl);
    for (int k = 0; k < n; ++k) t[k] = tl[k];
  }
  __syncthreads();
  double acc = 0.0;
  if (c.side == 0) {
    const double* g = c.G + (int64_t)c.ra * n * o;
#pragma unroll 4
    for (int e = threadIdx.x; e < c.ra * n; e += 256) {
      const int k = e / c.ra;
      acc = fma(c.x[e - k * c.ra] * t[k], g[e], acc);
    }
  } else {
    const double* g = c.G + o;
#pragma unroll 4
    for (int e = threadIdx.x; e < n * c.rb; e += 256) {
      const int q = e / n;
      acc = fma(t[e - q * n] * c.x[q], g[(int64_t)c.ra * e], acc);
    }
  }
  acc = warp_sum_d(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) acc += red[i];
    c.out[o] = acc;
  }
}

// out[i] = x_i . y_i (r_i values), up to three dot products, one block each
struct Dots {
  const double *x[3], *y[3];
  int r[3];
};
__global__ void __launch_bounds__(256) dots(Dots d, double* __restrict__ out) {
  __shared__ double red[8];
  const int i = blockIdx.x;
  double acc = 0.0;
  for (int k = threadIdx.x; k < d.r[i]; k += 256) acc = fma(d.x[i][k], d.y[i][k], acc);
  acc = warp_sum_d(acc);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) acc += red[k];
    out[i] = acc;
  }
}

// q[k] = sum_o Gs[k + K o] g[o]  (oriented core K x R_out, column-major): 32 values of k a block, the
// warps taking every eighth o, added in a fixed order
template <typename T>
__global__ void __launch_bounds__(256) core_times_vec(const T* __restrict__ Gs, int K, int R, const double* __restrict__ g,
                                                      T* __restrict__ q) {
  __shared__ double red[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + lane;
  double acc = 0.0;
  if (k < K)
    for (int o = w; o < R; o += 8) acc = fma((double)Gs[k + (int64_t)K * o], g[o], acc);
  red[w][lane] = acc;
  __syncthreads();
  if (w == 0 && k < K) {
    for (int i = 1; i < 8; ++i) acc += red[i][lane];
    q[k] = (T)acc;
  }
}

// Q[p, k] = sum_o Gbar[p, o] Gs[k + K o]  (Gbar: N x R row-major; Q: N x K row-major).
// 64 x 64 output tiles, 16-wide reduction chunks, 4 x 4 register tiles.
template <typename T>
__global__ void __launch_bounds__(256) gemm_gbar_core(const T* __restrict__ Gbar, const T* __restrict__ Gs,
                                                      int64_t N, int R, int K, T* __restrict__ Q) {
  __shared__ T As[16][65];
  __shared__ T Bs[16][65];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int64_t p0 = (int64_t)blockIdx.y * 64;
  const int k0 = blockIdx.x * 64;
  T acc[4][4] = {};
  for (int o0 = 0; o0 < R; o0 += 16) {
    for (int e = threadIdx.x; e < 64 * 16; e += 256) {
      const int pp = e / 16, oo = e % 16;
      const int64_t p = p0 + pp;
      As[oo][pp] = (p < N && o0 + oo < R) ? Gbar[p * R + o0 + oo] : T(0);
      const int kk = e % 64, o2 = e / 64;
      Bs[o2][kk] = (k0 + kk < K && o0 + o2 < R) ? Gs[(k0 + kk) + (int64_t)K * (o0 + o2)] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int oo = 0; oo < 16; ++oo) {
      T av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = As[oo][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = Bs[oo][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t p = p0 + ty * 4 + i;
    if (p >= N) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int k = k0 + tx * 4 + j;
      if (k < K) Q[p * K + k] = acc[i][j];
    }
  }
}

// Reverse step of the chain for one point per warp (see the file comment). Q is either the
// full N x K matrix (qvec == nullptr) or rank one: Q[p, k] = w[p] qvec[k].
template <typename T>
__global__ void __launch_bounds__(256) chain_back_step(const T* __restrict__ X, int d, int coord, double lo,
                                                       double hi, int n, int64_t N, int R_in,
                                                       const T* __restrict__ S_in, const T* __restrict__ Q,
                                                       const T* __restrict__ w, const T* __restrict__ qvec,
                                                       T* __restrict__ gbar_in, T* __restrict__ dX) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  T* db = reinterpret_cast<T*>(smem_raw) + (size_t)wib * (PTTK_MAX_N + R_in);  // dB[j], gbar[a]
  T* gb = db + PTTK_MAX_N;
  const int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + wib;
  if (p >= N) return;
  const double x = (double)X[p * d + coord];
  const double xh = (2.0 * x - lo - hi) / (lo - hi);
  for (int j = lane; j < PTTK_MAX_N; j += 32) db[j] = T(0);
  for (int a = lane; a < R_in; a += 32) gb[a] = T(0);
  __syncwarp();
  const int K = n * R_in;
  const T wp = qvec ? w[p] : T(0);
  for (int k = lane; k < K; k += 32) {
    const int j = k / R_in, a = k - j * R_in;
    const T qv = qvec ? wp * qvec[k] : Q[p * K + k];
    const T s = S_in ? S_in[p * R_in + a] : T(1);
    // T_j(xh) directly (cos form is avoided: the three-term recurrence below is per lane)
    double t0 = 1.0, t1 = xh, tj = 1.0;
    for (int m = 0; m <= j; ++m) {
      if (m == 0) tj = 1.0;
      else if (m == 1) tj = xh;
      else {
        const double t2 = 2.0 * xh * t1 - t0;
        t0 = t1;
        t1 = t2;
        tj = t2;
      }
    }
    atomicAdd(&db[j], s * qv);
    if (gbar_in) atomicAdd(&gb[a], (T)tj * qv);
  }
  __syncwarp();
  if (gbar_in)
    for (int a = lane; a < R_in; a += 32) gbar_in[p * R_in + a] = gb[a];
  if (lane == 0) {
    double td[PTTK_MAX_N];
    cheb_row(xh, n, true, 2.0 / (lo - hi), td);
    double acc = 0.0;
    for (int j = 0; j < n; ++j) acc = fma((double)db[j], td[j], acc);
    dX[p * d + coord] = (T)acc;
  }
}

// ---------------- reverse pass in one kernel ----------------------------------------------------
// dL/dX of the source points, one thread per point, nothing per point in memory but X, w and dX.
// With q[b + R_2 j] = (G_d^{2} g)[b, j] and w_p:
//   S_1 = B_1 G_1, S_2[b] = sum_{a,j} S_1[a] T_j(x_2) G_2[a, j, b]               (forward again)
//   e_j = sum_b S_2[b] q[b, j],  dL/dx_3 = w sum_j T_j'(x_3) e_j,  gbar_2[b] = w sum_j T_j(x_3) q[b, j]
//   Q[a, j] = sum_b gbar_2[b] G_2[a, j, b],  dL/dx_2 = sum_{a,j} S_1[a] T_j'(x_2) Q[a, j],
//   gbar_1[a] = sum_j T_j(x_2) Q[a, j],  dL/dx_1 = sum_{a,j} gbar_1[a] G_1[j, a] T_j'(x_1)
// (d = 2 lacks the middle step, d = 1 has the last alone.) The rows G_2[a, j, :] sit in shared memory,
// read as broadcasts; S_2 and gbar_2 (RB values, R_2 padded) in registers; the scalars that the loops
// index (T_j(x_2), the sums over a of S_1 Q, S_1, gbar_1) in shared memory, one column per thread. About
// 11k FMAs a point at ranks 9, 44: at N = 500k, n = 12 the separate kernels (S_1, S_2, Q and gbar
// in memory, shared-memory atomics per term) took 16.4 ms, this one 0.525 ms with scalar FP32 FMAs and 0.46 ms
// with the two-wide ones. What bounds it: issue, and the FP64 pipe for the bases.
// The bases are formed in FP64 and rounded to T; the last sum of each derivative, over T_j', is in FP64 (T_j' and the terms
// unrounded), as it is in the separate kernels.
constexpr int AF_THREADS = 128;

struct AdjArgs {
  int d, n, r1, r2;
  double lo[3], hi[3];
  int coord[3];
  const void* g1;  // oriented cores, column-major (R_in x n x R_out)
  const void* g2;
  const void* q;   // (R_in of the last step) x n, column-major
};

// T_j(x) (VALS) and T_j'(x) dxhat/dx = j U_{j-1}(x) dxhat/dx (DERIVS; else 0), j < n, handed to f(j, t, dt)
template <bool VALS, bool DERIVS, typename F>
__device__ __forceinline__ void cheb_each(double x, double lo, double hi, int n, F&& f) {
  const double xh = (2.0 * x - lo - hi) / (lo - hi), sc = 2.0 / (lo - hi), x2 = 2.0 * xh;
  double t0 = 1.0, t1 = xh, u0 = 0.0, u1 = sc, k = 1.0;
  f(0, 1.0, 0.0);
  for (int j = 1; j < n; ++j) {
    f(j, VALS ? t1 : 0.0, DERIVS ? k * u1 : 0.0);
    if (VALS) {
      const double t2 = fma(x2, t1, -t0);
      t0 = t1;
      t1 = t2;
    }
    if (DERIVS) {
      const double u2 = fma(x2, u1, -u0);
      u0 = u1;
      u1 = u2;
      k += 1.0;
    }
  }
}

template <typename T>
size_t adj_smem(int d, int n, int r1, int rb) {
  // G_1 (n x r1), q (n x rlast), G_2 (r1 n x rb), then per thread T_2, E_2 (n each), S_1, gbar_1 (r1 each)
  const size_t shared = (size_t)n * r1 + (size_t)n * (d == 3 ? rb : d == 2 ? r1 : 1) + (d == 3 ? (size_t)r1 * n * rb : 0);
  const size_t per = (size_t)2 * n + 2 * r1;
  return sizeof(T) * ((shared + 3) / 4 * 4 + per * AF_THREADS);
}

// acc[b] = m x[b] + acc[b], b < B (even), in FP32 by the two-wide instructions: half as many to issue, each half
// rounding as fmaf does
template <int B>
__device__ __forceinline__ void axpy(float m, const float* x, float* acc) {
  uint64_t mm;
  asm("mov.b64 %0, {%1, %1};" : "=l"(mm) : "f"(m));
#pragma unroll
  for (int b = 0; b < B; b += 2) {
    uint64_t y, z;
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(x[b]), "f"(x[b + 1]));
    asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(acc[b]), "f"(acc[b + 1]));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(z) : "l"(mm), "l"(y));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[b]), "=f"(acc[b + 1]) : "l"(z));
  }
}
template <int B>
__device__ __forceinline__ void axpy(double m, const double* x, double* acc) {
#pragma unroll
  for (int b = 0; b < B; ++b) acc[b] = fma(m, x[b], acc[b]);
}
// sum of x[b] y[b], b < B (a multiple of 4), in four partial sums
template <int B>
__device__ __forceinline__ float dot4(const float* x, const float* y) {
  uint64_t e[2] = {0, 0};
#pragma unroll
  for (int b = 0; b < B; b += 2) {
    uint64_t u, v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(u) : "f"(x[b]), "f"(x[b + 1]));
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(y[b]), "f"(y[b + 1]));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(e[(b >> 1) & 1]) : "l"(u), "l"(v));
  }
  float e0, e1, e2, e3;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(e0), "=f"(e1) : "l"(e[0]));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(e2), "=f"(e3) : "l"(e[1]));
  return (e0 + e1) + (e2 + e3);
}
template <int B>
__device__ __forceinline__ double dot4(const double* x, const double* y) {
  double e[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int b = 0; b < B; ++b) e[b & 3] = fma(x[b], y[b], e[b & 3]);
  return (e[0] + e[1]) + (e[2] + e[3]);
}

template <typename T, int D, int RB>
__global__ void __launch_bounds__(AF_THREADS) adj_reverse_kernel(AdjArgs a, const T* __restrict__ X, int64_t N,
                                                                 const T* __restrict__ w, T* __restrict__ dX) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int n = a.n, r1 = a.r1, tid = threadIdx.x;
  // rows of the last step's input: S_2 (d = 3, padded), S_1 (d = 2), 1 (d = 1)
  const int rl = D == 3 ? RB : D == 2 ? r1 : 1;
  T* G2 = reinterpret_cast<T*>(smem_raw);                 // [a][j][RB]
  T* q = G2 + (D == 3 ? (size_t)r1 * n * RB : 0);         // [j][rl]
  T* G1 = q + (size_t)n * rl;                             // [a][j]
  const size_t shared = (size_t)n * r1 + (size_t)n * rl + (D == 3 ? (size_t)r1 * n * RB : 0);
  T* priv = reinterpret_cast<T*>(smem_raw) + (shared + 3) / 4 * 4 + tid;
  T* T2 = priv;                          // [j] at stride AF_THREADS
  T* E2 = T2 + n * AF_THREADS;           // [j]: sum over a of S_1[a] Q[a, j]
  T* S1 = E2 + n * AF_THREADS;
  T* B1 = S1 + r1 * AF_THREADS;
  const int rlast = D == 3 ? a.r2 : D == 2 ? r1 : 1;
  if (D == 3)
    for (int e = tid; e < r1 * n * RB; e += AF_THREADS) {
      const int b = e % RB, aj = e / RB, j = aj % n, al = aj / n;
      G2[e] = b < a.r2 ? static_cast<const T*>(a.g2)[al + (size_t)r1 * (j + (size_t)n * b)] : T(0);
    }
  for (int e = tid; e < n * rl; e += AF_THREADS) {
    const int b = e % rl, j = e / rl;
    q[e] = b < rlast ? static_cast<const T*>(a.q)[b + (size_t)rlast * j] : T(0);
  }
  if (D >= 2)
    for (int e = tid; e < n * r1; e += AF_THREADS) {
      const int j = e % n, al = e / n;
      G1[e] = static_cast<const T*>(a.g1)[j + (size_t)n * al];
    }
  __syncthreads();
  for (int64_t p = (int64_t)blockIdx.x * AF_THREADS + tid; p < N; p += (int64_t)gridDim.x * AF_THREADS) {
    const T wp = w[p];
    double x[D];
#pragma unroll
    for (int i = 0; i < D; ++i) x[i] = (double)X[p * D + a.coord[i]];
    if constexpr (D == 1) {
      double acc = 0.0;
      cheb_each<false, true>(x[0], a.lo[0], a.hi[0], n, [&](int j, double, double dt) { acc = fma(dt, widen(q[j]), acc); });
      dX[p] = (T)(acc * widen(wp));
    } else {
      // S_1
      for (int al = 0; al < r1; ++al) S1[al * AF_THREADS] = T(0);
      cheb_each<true, false>(x[0], a.lo[0], a.hi[0], n, [&](int j, double t, double) {
        const T tj = (T)t;
        for (int al = 0; al < r1; ++al) S1[al * AF_THREADS] = fma(tj, G1[al * n + j], S1[al * AF_THREADS]);
      });
      if constexpr (D == 3) {
        cheb_each<true, false>(x[1], a.lo[1], a.hi[1], n, [&](int j, double t, double) {
          T2[j * AF_THREADS] = (T)t;
          E2[j * AF_THREADS] = T(0);
        });
        T s2[RB], gb[RB];
#pragma unroll
        for (int b = 0; b < RB; ++b) s2[b] = gb[b] = T(0);
        for (int al = 0; al < r1; ++al) {
          const T sa = S1[al * AF_THREADS];
          const T* row = G2 + (size_t)al * n * RB;
          for (int j = 0; j < n; ++j, row += RB) {
            axpy<RB>(sa * T2[j * AF_THREADS], row, s2);
          }
        }
        double dx3 = 0.0, dx2 = 0.0;
        cheb_each<true, true>(x[2], a.lo[2], a.hi[2], n, [&](int j, double t, double dt) {
          const T tj = (T)t * wp;
          const T* row = q + j * RB;
          axpy<RB>(tj, row, gb);
          dx3 = fma(dt, widen(dot4<RB>(s2, row)), dx3);
        });
        for (int al = 0; al < r1; ++al) {
          const T sa = S1[al * AF_THREADS];
          const T* row = G2 + (size_t)al * n * RB;
          T g1a = T(0);
          for (int j = 0; j < n; ++j, row += RB) {
            const T qv = dot4<RB>(gb, row);
            E2[j * AF_THREADS] = fma(sa, qv, E2[j * AF_THREADS]);
            g1a = fma(T2[j * AF_THREADS], qv, g1a);
          }
          B1[al * AF_THREADS] = g1a;
        }
        cheb_each<false, true>(x[1], a.lo[1], a.hi[1], n,
                               [&](int j, double, double dt) { dx2 = fma(dt, widen(E2[j * AF_THREADS]), dx2); });
        dX[p * D + a.coord[2]] = (T)(dx3 * widen(wp));
        dX[p * D + a.coord[1]] = (T)dx2;
      } else {
        for (int al = 0; al < r1; ++al) B1[al * AF_THREADS] = T(0);
        double dx2 = 0.0;
        cheb_each<true, true>(x[1], a.lo[1], a.hi[1], n, [&](int j, double t, double dt) {
          const T tj = (T)t * wp;
          const T* row = q + j * r1;
          T e = T(0);
          for (int al = 0; al < r1; ++al) {
            B1[al * AF_THREADS] = fma(tj, row[al], B1[al * AF_THREADS]);
            e = fma(S1[al * AF_THREADS], row[al], e);
          }
          dx2 = fma(dt, widen(e), dx2);
        });
        dX[p * D + a.coord[1]] = (T)(dx2 * widen(wp));
      }
      double dx1 = 0.0;
      cheb_each<false, true>(x[0], a.lo[0], a.hi[0], n, [&](int j, double, double dt) {
        T e = T(0);
        for (int al = 0; al < r1; ++al) e = fma(B1[al * AF_THREADS], G1[al * n + j], e);
        dx1 = fma(dt, widen(e), dx1);
      });
      dX[p * D + a.coord[0]] = (T)dx1;
    }
  }
}

template <typename T, int D, int RB>
pttk_status launch_adj(const AdjArgs& a, const T* X, int64_t N, const T* w, T* dX, cudaStream_t s) {
  auto kfn = adj_reverse_kernel<T, D, RB>;
  const size_t smem = adj_smem<T>(D, a.n, a.r1, RB);
  PTTK_CUDA(allow_smem((const void*)kfn));
  int per_sm = 1;
  PTTK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, AF_THREADS, smem));
  const int64_t blocks = std::min<int64_t>((N + AF_THREADS - 1) / AF_THREADS, (int64_t)sm_count() * std::max(per_sm, 1));
  kfn<<<(unsigned)blocks, AF_THREADS, smem, s>>>(a, X, N, w, dX);
  pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

// Padded R_2 of the one-kernel reverse pass; 0 where its registers (R_2 <= 64) or shared memory do not
// hold the ranks (the separate kernels then take the call).
template <typename T>
int adj_fused_rb(int d, int n, int r1, int r2) {
  const int rb = d < 3 ? 16 : r2 <= 16 ? 16 : r2 <= 32 ? 32 : r2 <= 48 ? 48 : r2 <= 64 ? 64 : 0;
  return rb && adj_smem<T>(d, n, r1, rb) <= 220 * 1024 ? rb : 0;
}

template <typename T>
pttk_status adj_reverse(int rb, const AdjArgs& a, const T* X, int64_t N, const T* w, T* dX, cudaStream_t s) {
  if (a.d == 1) return launch_adj<T, 1, 16>(a, X, N, w, dX, s);
  if (a.d == 2) return launch_adj<T, 2, 16>(a, X, N, w, dX, s);
  switch (rb) {
    case 16: return launch_adj<T, 3, 16>(a, X, N, w, dX, s);
    case 32: return launch_adj<T, 3, 32>(a, X, N, w, dX, s);
    case 48: return launch_adj<T, 3, 48>(a, X, N, w, dX, s);
    default: return launch_adj<T, 3, 64>(a, X, N, w, dX, s);
  }
}

template <typename T>
pttk_status weighted_sum(const T* A, const T* w, int64_t N, int r, double* out, double* partial, int nparts,
                         cudaStream_t s) {
  if (N == 0) {
    PTTK_CUDA(cudaMemsetAsync(out, 0, sizeof(double) * r, s));
    return PTTK_OK;
  }
  if (r % 4 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0) weighted_colsum<T, 4><<<nparts, 256, 0, s>>>(A, w, N, r, partial);
  else weighted_colsum<T, 1><<<nparts, 256, 0, s>>>(A, w, N, r, partial);
  pttk::count_launch();
  sum_partials<<<r, 256, 0, s>>>(partial, 4 * nparts, r, out); pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

struct Scratch {
  std::vector<void*> ptrs;
  cudaStream_t s;
  ~Scratch() {
    for (void* p : ptrs) cudaFreeAsync(p, s);
  }
  template <typename T>
  pttk_status get(T** out, size_t elems) {
    void* p = nullptr;
    const cudaError_t e = ws_malloc(&p, std::max<size_t>(elems, 1) * sizeof(T), s);
    if (e != cudaSuccess) return cuda_error(e, "adjoint scratch");
    ptrs.push_back(p);
    *out = static_cast<T*>(p);
    return PTTK_OK;
  }
};

template <typename T>
pttk_status grad_typed(const pttk_tt* tt, const double* theta, const T* X, int64_t N_s, const T* Y, int64_t N_t,
                       const T* w, const T* z, pttk_prec prec, double* loss, double* dtheta, T* dX,
                       cudaStream_t s) {
  const int d = tt->d, dth = tt->dtheta, n = tt->n, D = tt->D;
  const int rs = tt->ranks[d], rt = tt->ranks[d + dth];
  const bool fp64 = sizeof(T) == 8;
  Scratch sc{{}, s};
  T *U, *V;
  double *a, *b, *g, *partial, *small;
  PTTK_TRY(sc.get(&U, (size_t)N_s * rs));
  PTTK_TRY(sc.get(&V, (size_t)N_t * rt));
  const int nparts = (int)std::max<int64_t>(1, std::min<int64_t>((std::max(N_s, N_t) + 255) / 256, sm_count() * 4));
  PTTK_TRY(sc.get(&partial, (size_t)4 * nparts * std::max(rs, rt)));
  PTTK_TRY(sc.get(&a, rs));
  PTTK_TRY(sc.get(&b, rt));
  PTTK_TRY(sc.get(&g, rs));
  int rmax = 1;
  for (int k = 0; k <= D; ++k) rmax = std::max(rmax, tt->ranks[k]);
  PTTK_TRY(sc.get(&small, (size_t)8 * rmax + 8));

  // forward: U, V in the requested form
  double th[PTTK_MAX_D];
  for (int j = 0; j < dth; ++j) {
    const double lo = tt->box[d + j][0], hi = tt->box[d + j][1];
    th[j] = (2.0 * theta[j] - lo - hi) / (lo - hi);
  }
  PTTK_TRY(point_domain_check(tt, X, N_s, Y, N_t, fp64, tt_status_word(tt), s));
  if (prec == PTTK_FP64 || prec == PTTK_FP32) {
    PTTK_TRY(factor_build_both(tt, X, N_s, Y, N_t, prec, U, V, s));
  } else {
    // the shared-memory kernel: the theta-gradient is an FP64 result of these factors, and their last
    // FP32 bits differ between the chain kernels
    PTTK_TRY(factor_build_tc(tt, tt_tc_cache(tt), reinterpret_cast<const float*>(X), N_s,
                             reinterpret_cast<const float*>(Y), N_t, prec, reinterpret_cast<float*>(U),
                             reinterpret_cast<float*>(V), tt_status_word(tt), kTcSharedA, s));
  }
  PTTK_TRY(weighted_sum<T>(U, w, N_s, rs, a, partial, nparts, s));
  PTTK_TRY(weighted_sum<T>(V, z, N_t, rt, b, partial, nparts, s));
  // g = H b, L = a^T H b and dL/dtheta_j through vectors only: with one parameter g = H_1 b, L = a . g,
  // u = H_1'^T a, dtheta = u . b; with two v = H_2 b, v' = H_2' b, u = H_1^T a, u' = H_1'^T a, g = H_1 v,
  // L = u . v, dtheta = (u' . v, u . v').
  double *u = small + 8, *u1 = u + rmax, *v = u1 + rmax, *v1 = v + rmax;
  Dots dt{};
  int ndots = 1;
  if (dth == 0) {
    PTTK_CUDA(cudaMemcpyAsync(g, b, sizeof(double) * rs, cudaMemcpyDeviceToDevice, s));
    dt = Dots{{a}, {g}, {rs}};
  } else {
    const double* G1 = tt->cores64 + tt->core_off[d];
    const int r0 = tt->ranks[d], r1 = tt->ranks[d + 1], r2 = dth == 2 ? tt->ranks[d + 2] : 0;
    const double sc1 = 2.0 / (tt->box[d][0] - tt->box[d][1]);
    auto grid = [&](int count) { return dim3((unsigned)rmax, (unsigned)count); };
    if (dth == 1) {
      CoreVecs cv{{{G1, b, g, th[0], 1.0, r0, r1, 1, 0}, {G1, a, u1, th[0], sc1, r0, r1, 0, 1}}};
      core_vecs<<<grid(2), 256, 0, s>>>(cv, n); pttk::count_launch();
      dt = Dots{{a, u1}, {g, b}, {r0, r1}};
      ndots = 2;
    } else {
      const double* G2 = tt->cores64 + tt->core_off[d + 1];
      const double sc2 = 2.0 / (tt->box[d + 1][0] - tt->box[d + 1][1]);
      CoreVecs cv{{{G2, b, v, th[1], 1.0, r1, r2, 1, 0}, {G2, b, v1, th[1], sc2, r1, r2, 1, 1},
                   {G1, a, u, th[0], 1.0, r0, r1, 0, 0}, {G1, a, u1, th[0], sc1, r0, r1, 0, 1}}};
      core_vecs<<<grid(4), 256, 0, s>>>(cv, n); pttk::count_launch();
      CoreVecs cg{{{G1, v, g, th[0], 1.0, r0, r1, 1, 0}}};
      core_vecs<<<grid(1), 256, 0, s>>>(cg, n); pttk::count_launch();
      dt = Dots{{u, u1, u}, {v, v, v1}, {r1, r1, r1}};
      ndots = 3;
    }
  }
  dots<<<ndots, 256, 0, s>>>(dt, small); pttk::count_launch();

  // dL/dX by the reverse pass (SIMT, in the precision of X)
  if (dX && N_s > 0) {
    PTTK_PROF("adjoint", s);
    // last step: rank-one adjoint w_p g
    int rin, rout, coord;
    oriented_core_dims(tt, true, d - 1, &rin, &rout, &coord);
    const T* Gs_last = static_cast<const T*>(oriented_core_ptr(tt, true, d - 1, fp64));
    T* q;
    PTTK_TRY(sc.get(&q, (size_t)n * rin));
    core_times_vec<T><<<(unsigned)((n * rin + 31) / 32), 256, 0, s>>>(Gs_last, n * rin, rout, g, q); pttk::count_launch();
    const int rb = adj_fused_rb<T>(d, n, d > 1 ? tt->ranks[1] : 1, d > 2 ? tt->ranks[2] : 1);
    if (rb) {
      AdjArgs ar{};
      ar.d = d;
      ar.n = n;
      ar.r1 = d > 1 ? tt->ranks[1] : 1;
      ar.r2 = d > 2 ? tt->ranks[2] : 1;
      for (int i = 0; i < d; ++i) {
        int ri, ro;
        oriented_core_dims(tt, true, i, &ri, &ro, &ar.coord[i]);
        ar.lo[i] = tt->box[ar.coord[i]][0];
        ar.hi[i] = tt->box[ar.coord[i]][1];
      }
      ar.g1 = oriented_core_ptr(tt, true, 0, fp64);
      ar.g2 = d > 2 ? oriented_core_ptr(tt, true, 1, fp64) : nullptr;
      ar.q = q;
      PTTK_TRY(adj_reverse<T>(rb, ar, X, N_s, w, dX, s));
    } else {
      const pttk_prec simt = fp64 ? PTTK_FP64 : PTTK_FP32;
      std::vector<T*> Sbuf(d, nullptr);  // Sbuf[i] = S_i (N x r_i), i = 1..d-1
      for (int i = 1; i < d; ++i) {
        PTTK_TRY(sc.get(&Sbuf[i], (size_t)N_s * tt->ranks[i]));
        PTTK_TRY(factor_build_run(tt, true, X, N_s, simt, Sbuf[i], s, i));
      }
      T *gbar = nullptr, *gnext = nullptr, *Q = nullptr;
      size_t qmax = 0;
      for (int i = 0; i < d - 1; ++i) qmax = std::max<size_t>(qmax, (size_t)n * tt->ranks[i]);
      if (d > 1) {
        PTTK_TRY(sc.get(&gbar, (size_t)N_s * rmax));
        PTTK_TRY(sc.get(&gnext, (size_t)N_s * rmax));
        PTTK_TRY(sc.get(&Q, (size_t)N_s * qmax));
      }
      for (int i = d - 1; i >= 0; --i) {
        oriented_core_dims(tt, true, i, &rin, &rout, &coord);
        const double lo = tt->box[coord][0], hi = tt->box[coord][1];
        const int K = n * rin;
        if (i < d - 1) {
          const T* Gs = static_cast<const T*>(oriented_core_ptr(tt, true, i, fp64));
          dim3 grid((unsigned)((K + 63) / 64), (unsigned)((N_s + 63) / 64));
          gemm_gbar_core<T><<<grid, 256, 0, s>>>(gbar, Gs, N_s, rout, K, Q); pttk::count_launch();
        }
        const size_t smem = sizeof(T) * 8 * (PTTK_MAX_N + rin);
        chain_back_step<T><<<(unsigned)((N_s + 7) / 8), 256, smem, s>>>(
            X, d, coord, lo, hi, n, N_s, rin, i > 0 ? Sbuf[i] : nullptr, i < d - 1 ? Q : nullptr, w,
            i == d - 1 ? q : nullptr, i > 0 ? gnext : nullptr, dX); pttk::count_launch();
        std::swap(gbar, gnext);
      }
    }
  }
  PTTK_CUDA(cudaGetLastError());
  double host[3] = {0, 0, 0};
  PTTK_CUDA(cudaMemcpyAsync(host, small, sizeof(double) * 3, cudaMemcpyDeviceToHost, s));
  PTTK_CUDA(cudaStreamSynchronize(s));
  if (loss) *loss = host[0];
  if (dtheta)
    for (int j = 0; j < dth; ++j) dtheta[j] = host[1 + j];
  return PTTK_OK;
}

}  // namespace
}  // namespace pttk

using namespace pttk;

extern "C" pttk_status pttk_grad(const pttk_tt* tt, const double* theta, const void* X, int64_t N_s, const void* Y,
                                 int64_t N_t, const void* w, const void* z, pttk_prec prec, double* loss,
                                 double* dtheta, void* dX, void* stream) {
  clear_error();
  if (!tt || !theta) return set_error(PTTK_EINVAL, "NULL argument");
  if (N_s < 0 || N_t < 0) return set_error(PTTK_EINVAL, "negative point count");
  if ((N_s > 0 && (!X || !w)) || (N_t > 0 && (!Y || !z))) return set_error(PTTK_EINVAL, "NULL point or weight buffer");
  if (prec < PTTK_FP64 || prec > PTTK_FP16X3) return set_error(PTTK_EINVAL, "unknown precision");
  for (int j = 0; j < tt->dtheta; ++j) {
    const double lo = tt->box[tt->d + j][0], hi = tt->box[tt->d + j][1];
    if (!(theta[j] >= lo - 1e-12 * (hi - lo) && theta[j] <= hi + 1e-12 * (hi - lo)))
      return set_error(PTTK_EDOMAIN, "theta outside its box");
  }
  for (int k = 0; k < tt->d; ++k)
    if (tt->ranks[k] > 4096) return set_error(PTTK_ENOTSUP, "adjoint: rank above 4096");
  cudaStream_t s = as_stream(stream);
  if (prec == PTTK_FP64)
    return grad_typed<double>(tt, theta, static_cast<const double*>(X), N_s, static_cast<const double*>(Y), N_t,
                              static_cast<const double*>(w), static_cast<const double*>(z), prec, loss, dtheta,
                              static_cast<double*>(dX), s);
  return grad_typed<float>(tt, theta, static_cast<const float*>(X), N_s, static_cast<const float*>(Y), N_t,
                           static_cast<const float*>(w), static_cast<const float*>(z), prec, loss, dtheta,
                           static_cast<float*>(dX), s);
}
