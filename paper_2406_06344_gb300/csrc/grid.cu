// Offline stage, Phase 1: the grid tensor of kernel values at the tensor Chebyshev nodes
// (Eq. mdc) and its per-mode Chebyshev transform C = M x_1 A x_2 A ... x_D A with
// A[k, i] = (c_k / n) T_k(zeta_i) (Eq. cheb_trans written for coefficients).
//
// Layout: C is column-major (i_1 fastest, Section 2.2). Pass 1 (grid_tile_kernel) gives
// each CTA one tile of the leading m1 modes (fixed trailing indices): threads evaluate the tile's
// entries into shared memory, the tile's modes are transformed there one fibre per thread (held in
// registers), and the tile leaves in a single coalesced write. The other modes are then transformed in
// place by one strided pass each (mode_transform_kernel), consecutive threads taking consecutive entries
// of the leading block so every load and store is coalesced.
//
// The FP64 pipe (2 operations per clock per SM) bounds all of it, so the work is cut in three ways:
//  - A[k, n-1-i] = (-1)^k A[k, i], so a fibre is split into its even and odd part first: n + n^2 / 2 operations
//    instead of n^2.
//  - Where source and target box have the same centre in dimension s, kappa(|x - y|) does not change when x_s
//    and y_s are both reflected: M[i_s, k_s] = M[n-1-i_s, n-1-k_s], and C is zero unless the indices of x_s and y_s
//    have the same parity. Only the first half of the x_s nodes is evaluated and carried (the "folded"
//    tensor, 2^-s of the entries for s such dimensions); expand_kernel makes the x_s transforms last, where the parity
//    of y_s's index is known, and writes C with exact zeros. (d = 3 boxes shifted along one axis: s = 2.)
//  - r is formed once per point pair and used for all length scales; the Bessel table is read by Horner's
//    rule, and the exponential is the table form of fexp.cuh.
// 12^8 entries, general-nu Matern, FP64: 131.6 -> 20.3 ms (FP32 5.9 -> 4.8).
#include <math.h>

#include <algorithm>
#include <cmath>

#include "fexp.cuh"
#include "kernels.cuh"
#include "pttk_internal.cuh"

namespace pttk {
namespace {

struct GridArgs {
  int kind, d, dtheta, D, n, m1;
  int64_t tile, ntiles;
  int parts;             // threads that share the length scales of one point pair (grid_tile_kernel)
  int direct;            // kappa_l for every entry: FP32, kernels without a fast form, and scales whose inverse overflows
  int ext[PTTK_MAX_D];   // carried extent of each mode: n, or (n + 1) / 2 for a folded source mode
  double lo[PTTK_MAX_D], hi[PTTK_MAX_D];
  // general-nu Matern, grid tile kernel: per nu node, G(z) = z^nu e^z K_nu(z) on [kv_zlo, kv_zhi]
  // in kv_P pieces (see KvTable); kv_P = 0: the quadrature for every entry
  const void* kv_tab;
  int kv_P;
  double kv_zlo, kv_zhi, kv_inv_zlo;
  float kv_inv_log2q;
};

// ---------------- general-nu Matern by table ------------------------------------------------
// The grid's entries take z = sqrt(2 nu) r / l over a known range (the node distances and the
// l and nu nodes), and only n values of nu. For each nu node, G(z) = z^nu e^z K_nu(z), which
// is smooth for z > 0 with its one singularity (a branch point) at z = 0, is tabulated once as
// piecewise Chebyshev series: pieces [a, 1.5 a] from kv_zlo up (geometric, so each piece sees
// the singularity at the same relative distance: its Bernstein ellipse has rho ~ 9.9, and
// degree 16 leaves a truncation error near 1e-17), each series of degree KV_DEG fitted at the
// piece's KV_DEG + 1 first-kind Chebyshev points from the quadrature kv_scaled and kept as a polynomial
// in t in [-1, 1] (the Chebyshev coefficients fall like 9.9^-k and the change of basis grows like 2^k, so no
// accuracy is lost). An entry then costs one exponential and Horner's rule: kappa = c_nu e^{-z} G(z). Against 30-digit values
// the table is within 2.4e-15 (relative) for z in [1e-3, 60], nu in {0.5, 1, 2, 2.5, 4}.
// Entries outside the table's range (z below 1e-3 when boxes overlap) take the quadrature.
constexpr int KV_DEG = 16;
constexpr int KV_STRIDE = KV_DEG + 3;  // per piece: mid, 1 / half-width, KV_DEG + 1 coefficients
constexpr double KV_Q = 1.5;
constexpr int KV_MAX_PIECES = 64;

// One block per nu node: the pieces' values at their Chebyshev points, the coefficients
// c_m = (2 / (KV_DEG + 1)) sum_k G(z_k) T_m(zeta_k) (c_0 halved), then the powers' coefficients; FP64 and an
// FP32 copy.
struct KvBasis {
  double t[KV_DEG + 1][KV_DEG + 1];  // t[k][q]: coefficient of t^q in T_k
};
__global__ void __launch_bounds__(256) kv_table_kernel(int n, int P, double zlo, double nu_lo, double nu_hi, KvBasis basis,
                                                       double* __restrict__ tab64, float* __restrict__ tab32) {
  __shared__ double stab[KV_TABLE];
  __shared__ double vals[KV_MAX_PIECES * (KV_DEG + 1)];
  const int inu = blockIdx.x;
  kv_table_fill<double>(stab);
  const double zn = cospi((2.0 * inu + 1.0) / (2.0 * n));
  const double nu = 0.5 * (nu_lo - nu_hi) * zn + 0.5 * (nu_lo + nu_hi);
  __syncthreads();
  for (int e = threadIdx.x; e < P * (KV_DEG + 1); e += blockDim.x) {
    const int p = e / (KV_DEG + 1), k = e % (KV_DEG + 1);
    const double a = zlo * pow(KV_Q, (double)p), b = a * KV_Q;
    const double z = 0.5 * (a + b) + 0.5 * (b - a) * cospi((2.0 * k + 1.0) / (2.0 * (KV_DEG + 1)));
    vals[e] = exp(nu * log(z)) * kv_scaled<double>(nu, z, stab);
  }
  __syncthreads();
  __shared__ double cheb[KV_MAX_PIECES * (KV_DEG + 1)];
  for (int e = threadIdx.x; e < P * (KV_DEG + 1); e += blockDim.x) {
    const int p = e / (KV_DEG + 1), mm = e % (KV_DEG + 1);
    double acc = 0.0;
    for (int k = 0; k <= KV_DEG; ++k)
      acc = fma(vals[p * (KV_DEG + 1) + k], cospi((double)mm * (2.0 * k + 1.0) / (2.0 * (KV_DEG + 1))), acc);
    cheb[e] = (mm == 0 ? 1.0 : 2.0) / (KV_DEG + 1) * acc;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < P * KV_STRIDE; e += blockDim.x) {
    const int p = e / KV_STRIDE, m = e % KV_STRIDE;
    const double a = zlo * pow(KV_Q, (double)p), b = a * KV_Q;
    double v;
    if (m == 0) {
      v = 0.5 * (a + b);
    } else if (m == 1) {
      v = 2.0 / (b - a);
    } else {
      // coefficient of t^q in sum_k c_k T_k(t)
      const int q = m - 2;
      v = 0.0;
      for (int k = KV_DEG - ((KV_DEG - q) & 1); k >= q; k -= 2) v = fma(basis.t[k][q], cheb[p * (KV_DEG + 1) + k], v);
    }
    tab64[((size_t)inu * P + p) * KV_STRIDE + m] = v;
    tab32[((size_t)inu * P + p) * KV_STRIDE + m] = (float)v;
  }
}

__device__ __forceinline__ double exp_neg(double z, const double* __restrict__ ftab) { return fexp_neg(z, ftab); }
__device__ __forceinline__ float exp_neg(float z, const float*) { return expf(-z); }

// The quadrature, out of line: entries outside the table's range are rare.
template <typename T>
__device__ __noinline__ T kappa_matern_nu_slow(T r2, T l, T nu, T cnu, T snu, const T* __restrict__ stab) {
  return kappa_matern_nu<T>(r2, l, nu, cnu, snu, stab);
}

// kappa of the general-nu Matern from the table of nu node `inu`, or by quadrature outside it.
template <typename T>
__device__ __forceinline__ T kappa_matern_nu_tab(const GridArgs& a, int inu, T r2, T r, T l, T invl, T nu, T cnu, T snu,
                                                 const T* __restrict__ stab, const T* __restrict__ ftab) {
  const T z = sizeof(T) == 8 ? snu * invl * r : snu * r / l;
  if (a.kv_P > 0 && z >= T(a.kv_zlo) && z <= T(a.kv_zhi)) {
    int p = (int)(__log2f((float)z * (float)a.kv_inv_zlo) * a.kv_inv_log2q);
    p = min(max(p, 0), a.kv_P - 1);
    const T* c = static_cast<const T*>(a.kv_tab) + ((size_t)inu * a.kv_P + p) * KV_STRIDE;
    const T t = (z - __ldg(c)) * __ldg(c + 1);
    T G = __ldg(c + 2 + KV_DEG);
#pragma unroll
    for (int k = KV_DEG - 1; k >= 0; --k) G = fma(G, t, __ldg(c + 2 + k));
    return cnu * exp_neg(z, ftab) * G;
  }
  return kappa_matern_nu_slow<T>(r2, l, nu, cnu, snu, stab);
}

// Four closed forms from r^2 and r = sqrt(r^2), in FP64 with the table exponential (GridArgs::direct is 0 for these alone).
__device__ __forceinline__ double kappa_r(int kind, double r2, double r, double l, double invl, const double* __restrict__ ftab) {
  switch (kind) {
    case K_GAUSS: return fexp_neg(r2 * invl * invl, ftab);
    case K_MATERN32: {
      const double q = 1.7320508075688772 * invl * r, e = fexp_neg(q, ftab);
      return fma(q, e, e);
    }
    case K_EXPONENTIAL: return fexp_neg(r * invl, ftab);
    case K_MATERN52: {
      const double q = 2.23606797749979 * invl * r;
      return fma(q * q, 1.0 / 3.0, 1.0 + q) * fexp_neg(q, ftab);
    }
    default: return kappa_l<double>(kind, r2, l);
  }
}
// never taken in FP32
__device__ __forceinline__ float kappa_r(int kind, float r2, float, float l, float, const float*) {
  return kappa_l<float>(kind, r2, l);
}

// Chebyshev node table and Matern-nu node constants in shared memory.
template <typename T>
__device__ void fill_tables(const GridArgs& a, T* eta, T* cnu, T* snu, T* stab) {
  const int n = a.n;
  for (int e = threadIdx.x; e < a.D * n; e += blockDim.x) {
    const int j = e / n, i = e % n;
    // zeta_i = cos((2i+1) pi / (2n)) (0-based i), eta = phi_[lo,hi](zeta), phi as printed
    const double z = cospi((2.0 * i + 1.0) / (2.0 * n));
    eta[e] = (T)(0.5 * (a.lo[j] - a.hi[j]) * z + 0.5 * (a.lo[j] + a.hi[j]));
  }
  if (a.kind == K_MATERN_NU) {
    const int jn = a.d + 1;  // theta = (l, nu): nu is mode d + 2 (0-based d + 1)
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const double z = cospi((2.0 * i + 1.0) / (2.0 * n));
      const double nu = 0.5 * (a.lo[jn] - a.hi[jn]) * z + 0.5 * (a.lo[jn] + a.hi[jn]);
      cnu[i] = (T)(exp2(1.0 - nu) / tgamma(nu));
      snu[i] = (T)sqrt(2.0 * nu);
    }
    kv_table_fill<T>(stab);
  }
}

template <typename T>
__device__ __forceinline__ T eval_entry(const GridArgs& a, const int* idx, const T* eta,
                                        const T* cnu, const T* snu, const T* stab) {
  const int n = a.n;
  T r2 = T(0);
  for (int j = 0; j < a.d; ++j) {
    const T diff = eta[j * n + idx[j]] - eta[(a.d + a.dtheta + j) * n + idx[a.d + a.dtheta + j]];
    r2 += diff * diff;
  }
  const T l = a.dtheta > 0 ? eta[a.d * n + idx[a.d]] : T(1);
  if (a.kind == K_MATERN_NU) {
    const int inu = idx[a.d + 1];
    return kappa_matern_nu<T>(r2, l, eta[(a.d + 1) * n + inu], cnu[inu], snu[inu], stab);
  }
  return kappa_l<T>(a.kind, r2, l);
}

// Even and odd rows of the transform over the first half of the nodes, NBH = NB / 2 >= (n + 1) / 2 columns (zero
// past it): Ah[(k & 1) NBH^2 + (k >> 1) NBH + i] = A[k, i].
template <typename T, int NB>
__device__ __forceinline__ void fill_half(int n, T* Ah) {
  constexpr int NBH = NB / 2;
  for (int e = threadIdx.x; e < 2 * NBH * NBH; e += blockDim.x) {
    const int i = e % NBH, k = 2 * ((e / NBH) % NBH) + e / (NBH * NBH);
    double v = 0.0;
    if (i < (n + 1) / 2 && k < n) v = (k == 0 ? 1.0 : 2.0) / n * cospi((double)k * (2.0 * i + 1.0) / (2.0 * n));
    Ah[e] = (T)v;
  }
}

// Transform of one fibre (stride s) in place: E_i = x_i + x_{n-1-i}, O_i = x_i - x_{n-1-i} (the middle node of an
// odd n counts once, in E), y_{2m} = sum A[2m, i] E_i, y_{2m+1} = sum A[2m+1, i] O_i.
template <typename T, int NB>
__device__ __forceinline__ void transform_fibre(const T* __restrict__ Ah, int n, T* __restrict__ base, int64_t s) {
  constexpr int NBH = NB / 2;
  T ev[NBH], od[NBH];
#pragma unroll
  for (int i = 0; i < NBH; ++i) {
    const T lo = 2 * i + 1 <= n ? base[i * s] : T(0);
    const T hi = 2 * i + 1 < n ? base[(n - 1 - i) * s] : T(0);
    ev[i] = lo + hi;
    od[i] = 2 * i + 1 < n ? lo - hi : T(0);
  }
  // One pair of rows at a time: unrolled, the compiler keeps rows of Ah in registers across fibres and spills (20^6 general-nu
  // Matern 13.7 -> 12.9 ms in FP64, with the other changes 2.65 -> 1.22 ms in FP32).
#pragma unroll 1
  for (int m = 0; m < NBH; ++m) {
    T ye = T(0), yo = T(0);
#pragma unroll
    for (int i = 0; i < NBH; ++i) {
      ye = fma(Ah[m * NBH + i], ev[i], ye);
      yo = fma(Ah[NBH * NBH + m * NBH + i], od[i], yo);
    }
    if (2 * m < n) base[(2 * m) * s] = ye;
    if (2 * m + 1 < n) base[(2 * m + 1) * s] = yo;
  }
}

template <typename T, int NB>
__global__ void __launch_bounds__(512) grid_tile_kernel(GridArgs a, T* __restrict__ C) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tile = reinterpret_cast<T*>(smem_raw);
  T* eta = tile + a.tile;
  T* Ah = eta + a.D * a.n;
  T* cnu = Ah + 2 * (NB / 2) * (NB / 2);
  T* snu = cnu + a.n;
  T* ftab = snu + a.n;
  T* stab = ftab + FEXP_N;
  fill_tables<T>(a, eta, cnu, snu, stab);
  fill_half<T, NB>(a.n, Ah);
  if constexpr (sizeof(T) == 8)
    if (!a.direct) fexp_fill(ftab);
  __syncthreads();

  const int n = a.n, d = a.d, dth = a.dtheta, m1 = a.m1;
  // entries that differ in the first parameter (the length scale) alone share r: one thread evaluates
  // them all when that mode lies in the tile
  const bool inner = dth > 0 && m1 > d;
  const int nq = inner ? n : 1;
  int sx = 1;  // stride of the first parameter's mode in the tile
  for (int j = 0; j < min(m1, d); ++j) sx *= a.ext[j];
  const int tile_n = (int)a.tile, groups = tile_n / nq;
  const int per = (nq + a.parts - 1) / a.parts;
  for (int64_t t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
    int idx[PTTK_MAX_D];
    int64_t rem = t;
    for (int j = m1; j < a.D; ++j) {
      idx[j] = (int)(rem % a.ext[j]);
      rem /= a.ext[j];
    }
    for (int it = threadIdx.x; it < groups * a.parts; it += blockDim.x) {
      const int part = it / groups, g = it - part * groups;
      const int li0 = part * per, li1 = min(nq, li0 + per);
      int q = g;
      for (int j = 0; j < m1; ++j) {
        if (inner && j == d) continue;
        const int next = q / a.ext[j];
        idx[j] = q - next * a.ext[j];
        q = next;
      }
      T r2 = T(0);
      for (int j = 0; j < d; ++j) {
        const T diff = eta[j * n + idx[j]] - eta[(d + dth + j) * n + idx[d + dth + j]];
        r2 += diff * diff;
      }
      T* dst = tile + (inner ? g % sx + (g / sx) * sx * n + li0 * sx : g);
      const int l0 = inner ? 0 : dth > 0 ? idx[d] : 0;
      const int inu = dth > 1 ? idx[d + 1] : 0;
      if (a.direct) {
        for (int li = li0; li < li1; ++li, dst += sx) *dst = kappa_l<T>(a.kind, r2, dth > 0 ? eta[d * n + l0 + li] : T(1));
      } else {
        const T r = sqrt(r2);
        for (int li = li0; li < li1; ++li, dst += sx) {
          const T l = eta[d * n + l0 + li];
          const T invl = T(1) / l;
          *dst = a.kind == K_MATERN_NU
                     ? kappa_matern_nu_tab<T>(a, inu, r2, r, l, invl, eta[(d + 1) * n + inu], cnu[inu], snu[inu], stab, ftab)
                     : kappa_r(a.kind, r2, r, l, invl, ftab);
        }
      }
    }
    __syncthreads();
    // the tile's unfolded modes: one fibre per thread
    int st = 1;
    for (int j = 0; j < m1; st *= a.ext[j], ++j) {
      if (a.ext[j] != n) continue;
      const int nfib = tile_n / n;
      for (int f = threadIdx.x; f < nfib; f += blockDim.x) transform_fibre<T, NB>(Ah, n, tile + f % st + f / st * st * n, (int64_t)st);
      __syncthreads();
    }
    T* out = C + t * a.tile;
    for (int64_t e = threadIdx.x; e < a.tile; e += blockDim.x) out[e] = tile[e];
    __syncthreads();
  }
}

// In-place transform of one unfolded mode with stride s over the whole tensor.
template <typename T, int NB>
__global__ void __launch_bounds__(256) mode_transform_kernel(T* __restrict__ C, int n, int64_t s, int64_t nfib) {
  __shared__ T Ah[2 * (NB / 2) * (NB / 2)];
  fill_half<T, NB>(n, Ah);
  __syncthreads();
  for (int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; f < nfib;
       f += (int64_t)gridDim.x * blockDim.x)
    transform_fibre<T, NB>(Ah, n, C + f % s + f / s * s * n, s);
}

// The folded source modes' transforms and the write of C: for every trailing index (parameters and target
// modes) the block of the d source modes, `tin` values, goes through
//   y_h = sum_{i < (n+1)/2} w_i A[p_s + 2 h, i] x_i  (w_i = 2; 1 for the middle node of an odd n)
// along each folded mode s, p_s the parity of y_s's index, and leaves as n^d values, zero where a folded index has
// the other parity. `batch` trailing indices per block at a time.
template <typename T, int NB>
__global__ void __launch_bounds__(256) expand_kernel(GridArgs a, const T* __restrict__ F, int64_t tin, int64_t tout,
                                                     int64_t count, int batch, T* __restrict__ C) {
  constexpr int NBH = NB / 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw);  // batch x tin
  T* Ah = buf + (size_t)batch * tin;
  __shared__ int par[64][4];
  const int n = a.n, nh = (n + 1) / 2, d = a.d;
  fill_half<T, NB>(n, Ah);
  for (int64_t t0 = (int64_t)blockIdx.x * batch; t0 < count; t0 += (int64_t)gridDim.x * batch) {
    const int nb = (int)std::min<int64_t>(batch, count - t0);
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
      int64_t rem = t0 + b;
      for (int j = 0; j < a.dtheta; ++j) rem /= n;
      for (int j = 0; j < d; ++j) {
        par[b][j] = (int)(rem % n) & 1;
        rem /= n;
      }
    }
    for (int64_t e = threadIdx.x; e < nb * tin; e += blockDim.x) buf[e] = F[t0 * tin + e];
    __syncthreads();
    int64_t s = 1;
    for (int j = 0; j < d; s *= a.ext[j], ++j) {
      if (a.ext[j] == n) continue;
      const int64_t nfib = tin / nh;
      for (int64_t f = threadIdx.x; f < nb * nfib; f += blockDim.x) {
        const int b = (int)(f / nfib);
        const int64_t g = f % nfib;
        T* base = buf + b * tin + g % s + g / s * s * nh;
        const T* Ap = Ah + par[b][j] * NBH * NBH;
        T x[NBH];
#pragma unroll
        for (int i = 0; i < NBH; ++i) {
          const T v = i < nh ? base[i * s] : T(0);
          x[i] = 2 * i + 1 == n ? v : v + v;
        }
#pragma unroll 1
        for (int h = 0; h < NBH; ++h) {
          T y = T(0);
#pragma unroll
          for (int i = 0; i < NBH; ++i) y = fma(Ap[h * NBH + i], x[i], y);
          if (h < nh) base[h * s] = y;
        }
      }
      __syncthreads();
    }
    for (int64_t e = threadIdx.x; e < nb * tout; e += blockDim.x) {
      const int b = (int)(e / tout);
      int q = (int)(e % tout);
      int64_t src = 0, st = 1;
      bool keep = true;
      for (int j = 0; j < d; ++j) {
        const int i = q % n;
        q /= n;
        if (a.ext[j] == n) {
          src += i * st;
        } else {
          keep = keep && (i & 1) == par[b][j];
          src += (i >> 1) * st;
        }
        st *= a.ext[j];
      }
      C[t0 * tout + e] = keep ? buf[b * tin + src] : T(0);
    }
  }
}

// Extents of the modes (a source mode is folded where the boxes have the same centre, see the file comment)
// and the leading block of m1 modes held in shared memory.
void plan_tiles(GridArgs& a, bool fold, size_t elem) {
  const size_t budget = elem == 8 ? 170000 : 90000;
  for (int j = 0; j < a.D; ++j) a.ext[j] = a.n;
  for (int j = 0; fold && j < a.d; ++j)
    if (a.lo[j] + a.hi[j] == a.lo[a.d + a.dtheta + j] + a.hi[a.d + a.dtheta + j]) a.ext[j] = (a.n + 1) / 2;
  a.m1 = 1;
  a.tile = a.ext[0];
  a.ntiles = 1;
  for (int j = 1; j < a.D; ++j) a.ntiles *= a.ext[j];
  // A tile above 4096 entries only where that leaves every fourth SM one: a small grid in one tile is one block's work (32^3, boxes
  // equal, thin-plate spline FP64: 424 us in one tile, 155 in 32).
  while (a.m1 < a.D && (size_t)(a.tile * a.ext[a.m1]) * elem <= budget &&
         (a.tile * a.ext[a.m1] <= 4096 || a.ntiles / a.ext[a.m1] >= sm_count() / 4)) {
    a.ntiles /= a.ext[a.m1];
    a.tile *= a.ext[a.m1];
    ++a.m1;
  }
}

template <typename T, int NB>
pttk_status launch_all(GridArgs a, T* C, cudaStream_t st) {
  // folded tensor: in workspace memory, expanded into C at the end
  int64_t total = 1, folded = 1, tin = 1, tout = 1;
  for (int j = 0; j < a.D; ++j) {
    total *= a.n;
    folded *= a.ext[j];
    if (j < a.d) {
      tin *= a.ext[j];
      tout *= a.n;
    }
  }
  struct Fold {
    T* p = nullptr;
    cudaStream_t s;
    ~Fold() {
      if (p) cudaFreeAsync(p, s);
    }
  } fold{nullptr, st};
  T* F = C;
  if (folded != total) {
    const cudaError_t e = ws_malloc(&fold.p, sizeof(T) * (size_t)folded, st);
    if (e == cudaSuccess) {
      F = fold.p;
    } else if (e == cudaErrorMemoryAllocation) {  // no room beside C: the whole grid in place
      cudaGetLastError();
      fold.p = nullptr;
      plan_tiles(a, false, sizeof(T));
      folded = total;
    } else {
      PTTK_CUDA(e);
    }
  }
  const int threads = sizeof(T) == 8 ? 512 : 256;
  // The length scales of a point pair over `parts` threads: the fewest rounds of the block, each counted as its evaluations
  // and 0.4 for r (20^6 FP32: 400 pairs for 256 threads, 20 scales each, 78 % of the block busy; in 5 parts 98 %).
  a.parts = 1;
  if (a.dtheta > 0 && a.m1 > a.d) {
    double least = 0.0;
    for (int p = 1; p <= a.n; ++p) {
      const double cost = (double)((a.tile / a.n * p + threads - 1) / threads) * ((a.n + p - 1) / p + 0.4);
      if (p > 1 && cost >= least) continue;
      least = cost;
      a.parts = p;
    }
  }
  const size_t smem = sizeof(T) * (a.tile + (size_t)a.D * a.n + 2 * (NB / 2) * (NB / 2) + 2 * a.n + FEXP_N +
                                    (a.kind == K_MATERN_NU ? KV_TABLE : 0));
  auto kfn = grid_tile_kernel<T, NB>;
  PTTK_CUDA(allow_smem((const void*)kfn));
  int per_sm = 0;
  PTTK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, threads, smem));
  if (per_sm < 1) return set_error(PTTK_ENOTSUP, "grid tile does not fit on an SM");
  const int64_t grid = std::min<int64_t>(a.ntiles, (int64_t)sm_count() * per_sm);
  {
    PTTK_PROF("grid_tile", st);
    kfn<<<(unsigned)grid, threads, smem, st>>>(a, F); pttk::count_launch();
  }
  PTTK_CUDA(cudaGetLastError());
  const int64_t nfib = folded / a.n;
  int64_t s = a.tile;
  for (int j = a.m1; j < a.D; s *= a.ext[j], ++j) {
    if (a.ext[j] != a.n) continue;
    const int64_t blocks = std::min<int64_t>((nfib + 255) / 256, (int64_t)sm_count() * 8);
    PTTK_PROF("mode_transform", st);
    mode_transform_kernel<T, NB><<<(unsigned)blocks, 256, 0, st>>>(F, a.n, s, nfib); pttk::count_launch();
    PTTK_CUDA(cudaGetLastError());
  }
  if (folded != total) {
    const int64_t count = total / tout;
    // about 4096 values a block at a time, fewer where that leaves SMs without a block (9^6 FP64: 381 us with 18 indices a
    // block, 81 with 1)
    const int batch = (int)std::max<int64_t>(1, std::min<int64_t>({64, 4096 / tin, count / ((int64_t)sm_count() * 4)}));
    const size_t smem_e = sizeof(T) * ((size_t)batch * tin + 2 * (NB / 2) * (NB / 2));
    auto efn = expand_kernel<T, NB>;
    PTTK_CUDA(allow_smem((const void*)efn));
    const int64_t blocks = std::min<int64_t>((count + batch - 1) / batch, (int64_t)sm_count() * 16);
    PTTK_PROF("mode_transform", st);
    efn<<<(unsigned)blocks, 256, smem_e, st>>>(a, F, tin, tout, count, batch, C); pttk::count_launch();
    PTTK_CUDA(cudaGetLastError());
  }
  return PTTK_OK;
}

template <typename T>
pttk_status dispatch_nb(const GridArgs& a, T* C, cudaStream_t st) {
  const int nb = ((a.n + 3) / 4) * 4;
  switch (nb) {
    case 4: return launch_all<T, 4>(a, C, st);
    case 8: return launch_all<T, 8>(a, C, st);
    case 12: return launch_all<T, 12>(a, C, st);
    case 16: return launch_all<T, 16>(a, C, st);
    case 20: return launch_all<T, 20>(a, C, st);
    case 24: return launch_all<T, 24>(a, C, st);
    case 28: return launch_all<T, 28>(a, C, st);
    case 32: return launch_all<T, 32>(a, C, st);
  }
  return set_error(PTTK_EINVAL, "n out of range");
}

// Entries of the grid tensor M (Eq. mdc) at a list of multi-indices (the entry access the
// TT greedy-cross works from): out[e] = f_kappa(eta^(1)_{idx[e,0]}, ..., eta^(D)_{idx[e,D-1]}),
// idx row-major M x D. An index outside [0, n) gives NaN and records PTTK_EINVAL in *status;
// no node is read with it.
template <typename T>
__global__ void __launch_bounds__(256) entries_kernel(GridArgs a, const int* __restrict__ idx, int64_t M,
                                                      T* __restrict__ out, int* __restrict__ status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* eta = reinterpret_cast<T*>(smem_raw);
  T* cnu = eta + a.D * a.n;
  T* snu = cnu + a.n;
  T* stab = snu + a.n;
  fill_tables<T>(a, eta, cnu, snu, stab);
  __syncthreads();
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < M;
       e += (int64_t)gridDim.x * blockDim.x) {
    int row[PTTK_MAX_D];
    bool ok = true;
    for (int j = 0; j < a.D; ++j) {
      const int v = idx[e * a.D + j];
      ok = ok && v >= 0 && v < a.n;
      row[j] = ok ? v : 0;
    }
    if (!ok) {
      out[e] = T(NAN);
      atomicExch(status, (int)PTTK_EINVAL);
      continue;
    }
    out[e] = eval_entry<T>(a, row, eta, cnu, snu, stab);
  }
}

template <typename T>
pttk_status launch_entries(const GridArgs& a, const int* idx, int64_t M, T* out, int* status,
                           cudaStream_t st) {
  const size_t smem = sizeof(T) * ((size_t)a.D * a.n + 2 * a.n +
                                   (a.kind == K_MATERN_NU ? KV_TABLE : 0));
  auto kfn = entries_kernel<T>;
  PTTK_CUDA(allow_smem((const void*)kfn));
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((M + 255) / 256, (int64_t)sm_count() * 8));
  PTTK_PROF("grid_entries", st);
  kfn<<<(unsigned)blocks, 256, smem, st>>>(a, idx, M, out, status); pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

}  // namespace

pttk_status grid_entries_launch(int kernel, int d, int dtheta, int n, const double (*box)[2],
                                const int* idx, int64_t M, bool fp64, void* out, int* status,
                                cudaStream_t s) {
  if (M == 0) return PTTK_OK;
  GridArgs a{};
  a.kind = kernel;
  a.d = d;
  a.dtheta = dtheta;
  a.D = 2 * d + dtheta;
  a.n = n;
  for (int j = 0; j < a.D; ++j) {
    a.lo[j] = box[j][0];
    a.hi[j] = box[j][1];
  }
  if (fp64) return launch_entries<double>(a, idx, M, static_cast<double*>(out), status, s);
  return launch_entries<float>(a, idx, M, static_cast<float*>(out), status, s);
}

pttk_status grid_coeffs_launch(int kernel, int d, int dtheta, int n, const double (*box)[2],
                               bool fp64, void* C, cudaStream_t s) {
  GridArgs a{};
  a.kind = kernel;
  a.d = d;
  a.dtheta = dtheta;
  a.D = 2 * d + dtheta;
  a.n = n;
  for (int j = 0; j < a.D; ++j) {
    a.lo[j] = box[j][0];
    a.hi[j] = box[j][1];
  }
  const bool closed = kernel == K_GAUSS || kernel == K_MATERN32 || kernel == K_EXPONENTIAL || kernel == K_MATERN52;
  a.direct = kernel != K_MATERN_NU && !(closed && fp64 && std::isfinite(1.0 / a.lo[d]));
  plan_tiles(a, true, fp64 ? 8 : 4);
  // the per-nu tables live until the kernels that read them have run: released stream-ordered
  // on every return path
  struct Tables {
    double* t64 = nullptr;
    float* t32 = nullptr;
    cudaStream_t s;
    ~Tables() {
      if (t64) cudaFreeAsync(t64, s);
      if (t32) cudaFreeAsync(t32, s);
    }
  } tabs{nullptr, nullptr, s};
  double*& tab64 = tabs.t64;
  float*& tab32 = tabs.t32;
  if (kernel == K_MATERN_NU) {
    // the range of z = sqrt(2 nu) r / l over the grid's nodes
    auto node = [&](int j, int i) {
      const double z = cos((2.0 * i + 1.0) * 3.14159265358979323846 / (2.0 * n));
      return 0.5 * (a.lo[j] - a.hi[j]) * z + 0.5 * (a.lo[j] + a.hi[j]);
    };
    double r2min = 0.0, r2max = 0.0;
    for (int j = 0; j < d; ++j) {
      double dmin = INFINITY, dmax = 0.0;
      for (int i = 0; i < n; ++i)
        for (int k = 0; k < n; ++k) {
          const double df = fabs(node(j, i) - node(d + dtheta + j, k));
          dmin = std::min(dmin, df);
          dmax = std::max(dmax, df);
        }
      r2min += dmin * dmin;
      r2max += dmax * dmax;
    }
    double lmin = INFINITY, lmax = 0.0, numin = INFINITY, numax = 0.0;
    for (int i = 0; i < n; ++i) {
      lmin = std::min(lmin, node(d, i));
      lmax = std::max(lmax, node(d, i));
      numin = std::min(numin, node(d + 1, i));
      numax = std::max(numax, node(d + 1, i));
    }
    double zlo = std::max(sqrt(2.0 * numin) * sqrt(r2min) / lmax * (1.0 - 1e-12), 1e-3);
    const double zhi = std::min(sqrt(2.0 * numax) * sqrt(r2max) / lmin * (1.0 + 1e-12), 700.0);
    if (zhi > zlo) {
      int P = (int)ceil(log(zhi / zlo) / log(KV_Q));
      if (P > KV_MAX_PIECES) {
        P = KV_MAX_PIECES;
        zlo = zhi / pow(KV_Q, (double)P);
      }
      P = std::max(P, 1);
      const size_t cnt = (size_t)n * P * KV_STRIDE;
      PTTK_CUDA(ws_malloc(&tab64, sizeof(double) * cnt, s));
      PTTK_CUDA(ws_malloc(&tab32, sizeof(float) * cnt, s));
      KvBasis basis{};  // T_{k+1} = 2 t T_k - T_{k-1}, exact integers
      basis.t[0][0] = basis.t[1][1] = 1.0;
      for (int k = 2; k <= KV_DEG; ++k)
        for (int q = 0; q <= k; ++q) basis.t[k][q] = (q > 0 ? 2.0 * basis.t[k - 1][q - 1] : 0.0) - basis.t[k - 2][q];
      kv_table_kernel<<<n, 256, 0, s>>>(n, P, zlo, a.lo[d + 1], a.hi[d + 1], basis, tab64, tab32); pttk::count_launch();
      PTTK_CUDA(cudaGetLastError());
      a.kv_tab = fp64 ? static_cast<const void*>(tab64) : static_cast<const void*>(tab32);
      a.kv_P = P;
      a.kv_zlo = zlo;
      a.kv_zhi = zhi;
      a.kv_inv_zlo = 1.0 / zlo;
      a.kv_inv_log2q = (float)(1.0 / log2(KV_Q));
    }
  }
  return fp64 ? dispatch_nb<double>(a, static_cast<double*>(C), s) : dispatch_nb<float>(a, static_cast<float*>(C), s);
}

}  // namespace pttk
