// Offline stage, Phase 2 with TT-SVD (Section 2.3; Oseledets 2011, Algorithm 1) in place
// of TT greedy-cross, entirely in FP64 on the device.
//
// Step k (k = 1..D-1) works on the unfolding X (m x c, column-major, m = r_{k-1} n):
//   wide  (c >= m): W = X^T; R = qr_r(W) (Householder); one-sided Jacobi on R gives
//                   R V = U_R Sigma, so the left singular vectors of X are V. The core is
//                   G_k = V[:, top r] and the remainder X <- G_k^T X.
//   tall  (c <  m): R = qr_r(X); Jacobi on R gives Sigma and the right singular vectors V;
//                   Y = X V[:, top r] spans the top-r left singular subspace; a second
//                   Jacobi pass orthogonalises Y's columns (they are nearly orthogonal
//                   already) and G_k is Y with unit columns; X <- G_k^T X.
// In both cases G_k has orthonormal columns to working precision, so G_k G_k^T X is the
// orthogonal projection of X and the discarded part has norm sqrt(sum_{i>r} sigma_i^2).
// r_k is the smallest r >= 1 with that tail <= delta = tol / sqrt(D-1) ||C||_F (the
// threshold of Algorithm 1, TT-Round). QR first keeps singular values down to
// ~1e-16 ||X|| meaningful (a Gram-matrix route would lose everything below ~1e-8 ||X||).
//
// The QR (hh_kernel) and the Jacobi (jacobi_kernel) are cooperative launches whose blocks meet at grid
// barriers with bounded waits; every other kernel is a grid of independent blocks.
//
// Parity sectors. Where the boxes have a common centre in dimension s, C vanishes unless the indices of x_s
// and y_s have the same parity (grid.cu writes those zeros exactly; find_sectors looks for them in any
// C). Rows and columns of every unfolding then carry a charge, one bit per such dimension (the parity of
// the index of x_s or y_s among them), X is zero between rows and columns of different charge, and its SVD is
// the union of the SVDs of its 2^s diagonal blocks. Each step factors the blocks (in one batch of launches)
// and truncates their singular values together, so ranks and threshold are those of the whole unfolding.
// For s = 2 the QR and the Jacobi have a sixteenth of the operations. d = 3, 12^8: TT-SVD 0.90 s ->
// 0.16 s.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <numeric>
#include <vector>

#include "pttk_internal.cuh"

namespace pttk {
namespace {

constexpr int HU = 8;     // rows per lane per load batch in the Householder passes

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int THREADS>
__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (l < THREADS / 32) ? red[l] : 0.0;
    v = warp_sum(v);
  }
  __syncthreads();
  return v;  // valid in warp 0
}

// partial[b] = sum of squares of x over the block's grid-stride share
__global__ void __launch_bounds__(256) sumsq_kernel(const double* __restrict__ x, int64_t n,
                                                    double* __restrict__ partial) {
  __shared__ double red[8];
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    acc = fma(x[i], x[i], acc);
  acc = block_sum<256>(acc, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

__global__ void sum_kernel(const double* __restrict__ partial, int np, double* __restrict__ out) {
  __shared__ double red[8];
  double acc = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) acc += partial[i];
  acc = block_sum<256>(acc, red);
  if (threadIdx.x == 0) *out = acc;
}

// W (c x m, column-major) = (P X)^T for X m x c column-major, where row i of P X is row
// rowperm[i] of X (rowperm may be null: identity)
__global__ void transpose_kernel(const double* __restrict__ X, int64_t m, int64_t c,
                                 const int* __restrict__ rowperm, double* __restrict__ W) {
  __shared__ double t[32][33];
  const int64_t c0 = (int64_t)blockIdx.x * 32, m0 = (int64_t)blockIdx.y * 32;
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int64_t row = m0 + threadIdx.x, col = c0 + yy;
    if (row < m && col < c) t[yy][threadIdx.x] = X[(rowperm ? rowperm[row] : row) + col * m];
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < 32; yy += blockDim.y) {
    const int64_t row = c0 + threadIdx.x, col = m0 + yy;  // W[row, col] = X[col, row]
    if (row < c && col < m) W[row + col * c] = t[threadIdx.x][yy];
  }
}

// ---------------- Householder QR with column pivoting, truncated --------------------------
// A: M x N column-major (M >= N), overwritten. Step j picks, among the columns not yet
// factored, the one with the largest norm in rows j..M-1 (ties: lowest position), moves it to
// position j, and reflects it: x = A[j:M, p], beta = -sign(x_0) ||x||,
// v = [1; x_{1:}/(x_0 - beta)], tau = (beta - x_0) / beta, H_j = I - tau v v^T,
// H_j x = beta e_1 (LAPACK convention). The factorisation stops before step j as soon as
// the remaining block A[j:M, j:N] (the R22 of A P = Q [R11 R12; 0 R22]) has Frobenius norm
// <= `stop`: then A P = Q [R11 R12] + (a term of norm ||R22||_F), which is what the
// truncated SVD downstream needs, and k = j rows of R are kept.
//
// Columns are never moved: perm[l] is the physical column at position l (pivots in order, then the
// others), the reflector data of step j stays in physical column perm[j], and R is stored by physical
// column, Rp[i + N * perm[l]] = R[i, l]. The norm of every remaining column below the next diagonal
// row comes exactly from the update of the previous step (per row group, summed in a fixed order), so
// pivots and the stopping test use exact norms, not downdated ones.
//
// One cooperative launch per batch of matrices. A matrix has RG x CN blocks: in each step block (rg, cb) takes the rows
// of group rg and share cb of the columns left, 16 at a time (two per warp). A step is: dot products of the
// reflector with the block's columns (partial per row group), a barrier among the matrix's blocks, the update with the
// new norms, a barrier, and the pivot choice, which every block makes for itself from the same numbers. What
// bounds it: 3 FP64 FMAs per remaining element and step where the matrix is large, two barriers a step
// (about 5 us in all) where it is small. As five launches a step, the QRs of 20^5 took 15.8 ms,
// now 4.0 (with the sectors).
// The columns are dealt anew in each step: with a block keeping its columns for good, the warps whose columns were taken as
// pivots stood idle (20736 x 3696, 1350 steps: 827 ms; five launches a step 575; now 571). Large batches run three blocks an SM
// for the FP64 pipe (248832 x 756: 417 -> 402 ms), small ones two, since a barrier costs more with more blocks (3672 x 144: 3.5
// against 5.1 ms); the line, 8 million elements, lies between 7281 x 729 (23.6 against 27.1 ms) and 10008 x 1728
// (71.9 against 59.5). The former also pass 4096 rows of the reflector at a time instead of 1024 (417 against 438 ms, two blocks).
struct HHState {
  double tail2;  // ||R22||_F^2 at the stop (0 if every column was factored)
  int k;
};

struct alignas(128) GridSync {     // a barrier among the blocks of one matrix (zeroed before the launch)
  alignas(128) unsigned count;     // arrivals
  alignas(128) unsigned gen;       // generation (polled: its own line)
  alignas(128) int err;            // a barrier wait gave up
};

// Bounded barrier among `nblocks` blocks of a cooperative launch (so every block is resident): gives up
// after ~2 s (2^32 SM clocks) or once another block has given up; returns false then.
__device__ bool grid_barrier(GridSync* js, unsigned nblocks) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* vgen = &js->gen;
    volatile int* verr = &js->err;
    const unsigned gen = *vgen;
    __threadfence();
    int ok = 1;
    if (atomicAdd(&js->count, 1u) == nblocks - 1) {
      atomicExch(&js->count, 0u);
      __threadfence();
      atomicAdd(&js->gen, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == gen) {
        __nanosleep(32);
        if (*verr) {
          ok = 0;
          break;
        }
        if (clock64() - t0 > (4ll << 30)) {
          atomicExch(&js->err, 1);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    s_ok = ok && !*verr;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int MAX_JOBS = 8;        // matrices of one batch (2^3 sectors)
constexpr int QC = 16;             // columns of a block at a time: two per warp

struct QrJob {
  double* A;
  int64_t M;
  int N, rg, cn, block0;  // row groups, column sets, first block
  double stop2;
  double* Rp;             // N x N, zero
  int* perm;              // N
  double *part, *wpart;   // rg x N each
  double* xrow;           // N: the next diagonal row
  HHState* st;
  GridSync* sync;
};
struct QrBatch {
  QrJob j[MAX_JOBS];
  int count;
};

template <int PER_SM, int RC>  // RC: rows per pass of the reflector through shared memory
__global__ void __launch_bounds__(256, PER_SM) hh_kernel(QrBatch batch) {
  extern __shared__ unsigned mask[];  // bit p: column p not yet factored; then the columns left before each word
  __shared__ double v[RC];
  __shared__ double s_tot[8], s_max[8], s_x0, s_below;
  __shared__ int s_arg[8];
  int q = batch.count - 1;
  while ((int)blockIdx.x < batch.j[q].block0) --q;
  const QrJob& jb = batch.j[q];
  const int lb = (int)blockIdx.x - jb.block0, RG = jb.rg, CN = jb.cn, N = jb.N;
  const unsigned nblocks = (unsigned)(RG * CN);
  if (lb >= (int)nblocks) return;
  const int rg = lb % RG, cb = lb / RG;
  const int64_t M = jb.M, r_lo = M * rg / RG, r_hi = M * (rg + 1) / RG;
  double* __restrict__ A = jb.A;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = (N + 31) / 32;
  int* before = reinterpret_cast<int*>(mask + nw);
  for (int e = threadIdx.x; e < nw; e += 256) {
    mask[e] = 32 * e + 32 <= N ? 0xffffffffu : (1u << (N & 31)) - 1u;
    before[e] = 32 * e;
  }
  // physical column of the q-th one left, by a whole warp
  auto column = [&](int q) -> int {
    int w = -1;
    for (int base = 0; base < nw; base += 32) {
      const unsigned le = __ballot_sync(0xffffffffu, base + lane < nw && before[base + lane] <= q);
      w += __popc(le);
      if (le != 0xffffffffu) break;
    }
    const unsigned word = mask[w];
    const bool hit = (word >> lane & 1u) && __popc(word & ((1u << lane) - 1u)) == q - before[w];
    return 32 * w + __ffs(__ballot_sync(0xffffffffu, hit)) - 1;
  };
  // squares below the first row, and the first row
  for (int c0 = cb * QC; c0 < N; c0 += CN * QC)
    for (int c = 0; c < 2; ++c) {
      const int p = c0 + 2 * warp + c;
      if (p >= N) continue;
      const double* col = A + (int64_t)p * M;
      double acc = 0.0;
      for (int64_t i = std::max<int64_t>(r_lo, 1) + lane; i < r_hi; i += 32) acc = fma(col[i], col[i], acc);
      acc = warp_sum(acc);
      if (lane == 0) {
        jb.part[(int64_t)rg * N + p] = acc;
        if (r_lo == 0) jb.xrow[p] = col[0];
      }
    }
  if (!grid_barrier(jb.sync, nblocks)) return;
  for (int j = 0; j < N; ++j) {
    // pivot, stopping test and reflector of step j
    double tot = 0.0, best = -1.0;
    int arg = N;
    for (int p = threadIdx.x; p < N; p += 256) {
      if (!(mask[p >> 5] >> (p & 31) & 1u)) continue;
      double below = 0.0;
      for (int g = 0; g < RG; ++g) below += __ldcg(jb.part + (int64_t)g * N + p);
      const double x = __ldcg(jb.xrow + p);
      const double t = fma(x, x, below);
      tot += t;
      if (t > best) {  // strictly greater: the lowest column wins ties within a thread
        best = t;
        arg = p;
      }
    }
    // fixed-order reductions: the sum, and the largest with the lowest column on ties
    for (int o = 16; o; o >>= 1) {
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
      if (ob > best || (ob == best && oa < arg)) {
        best = ob;
        arg = oa;
      }
    }
    if (lane == 0) {
      s_tot[warp] = tot;
      s_max[warp] = best;
      s_arg[warp] = arg;
    }
    __syncthreads();
    tot = s_tot[0];
    best = s_max[0];
    arg = s_arg[0];
    for (int w = 1; w < 8; ++w) {
      tot += s_tot[w];
      if (s_max[w] > best || (s_max[w] == best && s_arg[w] < arg)) {
        best = s_max[w];
        arg = s_arg[w];
      }
    }
    if (j > 0 && tot <= jb.stop2) {
      if (lb == 0 && threadIdx.x == 0) {
        *jb.st = HHState{tot, j};
        int l = j;
        for (int p = 0; p < N; ++p)
          if (mask[p >> 5] >> (p & 31) & 1u) jb.perm[l++] = p;
      }
      return;
    }
    if (arg >= N) {  // only NaN columns are left: the lowest
      arg = 0;
      while (!(mask[arg >> 5] >> (arg & 31) & 1u)) ++arg;
    }
    const int pj = arg;
    if (threadIdx.x == 0) {
      double below = 0.0;
      for (int g = 0; g < RG; ++g) below += __ldcg(jb.part + (int64_t)g * N + pj);
      s_below = below;
      s_x0 = __ldcg(jb.xrow + pj);
    }
    __syncthreads();
    const double x0 = s_x0, acc2 = s_below;
    double beta = x0, scale = 0.0, tau = 0.0;
    if (acc2 > 0.0) {  // else nothing below the diagonal: no reflection
      const double nrm = hypot(x0, sqrt(acc2));
      beta = (x0 >= 0.0) ? -nrm : nrm;
      scale = 1.0 / (x0 - beta);
      tau = (beta - x0) / beta;
    }
    if (threadIdx.x == 0) mask[pj >> 5] &= ~(1u << (pj & 31));
    for (int e = (pj >> 5) + 1 + threadIdx.x; e < nw; e += 256) --before[e];
    if (lb == 0 && threadIdx.x == 0) {
      jb.perm[j] = pj;
      jb.Rp[j + (int64_t)pj * N] = beta;
    }
    if (j == N - 1) break;
    __syncthreads();
    const double* vj = A + (int64_t)pj * M;
    const int64_t b_lo = std::max<int64_t>(r_lo, j);
    // the reflector stays in shared memory between the two passes when the block has one set of columns and
    // at most RC rows
    const bool keep = N <= CN * QC && r_hi - b_lo <= RC;
    auto load_v = [&](int64_t lo, int rows) {
      __syncthreads();
      for (int t = threadIdx.x; t < rows; t += 256) v[t] = lo + t == j ? 1.0 : __ldcg(vj + lo + t) * scale;
      __syncthreads();
    };
    // this block's share of the columns left
    // (32 bits: R takes N^2 doubles, so N < 2^18, and there are a few hundred blocks)
    const unsigned left = (unsigned)(N - 1 - j);
    const int q_lo = (int)(left * (unsigned)cb / (unsigned)CN), q_hi = (int)(left * (unsigned)(cb + 1) / (unsigned)CN);
    int p0 = 0, p1 = 0;  // kept for the second pass where there is one set
    const bool one_set = q_hi - q_lo <= QC;
    for (int c0 = q_lo; c0 < q_hi; c0 += QC) {
      const bool l0 = c0 + warp < q_hi, l1 = c0 + warp + 8 < q_hi;
      p0 = l0 ? column(c0 + warp) : 0;
      p1 = l1 ? column(c0 + warp + 8) : 0;
      const double* ca = A + (int64_t)p0 * M;
      const double* cbp = A + (int64_t)p1 * M;
      double a0 = 0.0, a1 = 0.0;
      for (int64_t lo = b_lo; lo < r_hi; lo += RC) {
        const int rows = (int)std::min<int64_t>(RC, r_hi - lo);
        load_v(lo, rows);
        if (!l0) continue;
        for (int t0 = lane; t0 < rows; t0 += 32 * HU) {
          double x[HU], y[HU];  // all loads in flight before the arithmetic
#pragma unroll
          for (int u = 0; u < HU; ++u) {
            const bool in = t0 + 32 * u < rows;
            x[u] = in ? __ldcg(ca + lo + t0 + 32 * u) : 0.0;
            y[u] = in && l1 ? __ldcg(cbp + lo + t0 + 32 * u) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < HU; ++u) {
            const double vv = t0 + 32 * u < rows ? v[t0 + 32 * u] : 0.0;
            a0 = fma(vv, x[u], a0);
            a1 = fma(vv, y[u], a1);
          }
        }
      }
      a0 = warp_sum(a0);
      a1 = warp_sum(a1);
      if (lane == 0) {
        if (l0) jb.wpart[(int64_t)rg * N + p0] = a0;
        if (l1) jb.wpart[(int64_t)rg * N + p1] = a1;
      }
    }
    if (!grid_barrier(jb.sync, nblocks)) return;
    for (int c0 = q_lo; c0 < q_hi; c0 += QC) {
      const bool l0 = c0 + warp < q_hi, l1 = c0 + warp + 8 < q_hi;
      if (!one_set) {
        p0 = l0 ? column(c0 + warp) : 0;
        p1 = l1 ? column(c0 + warp + 8) : 0;
      }
      // w = tau sum over the row groups
      double w0 = 0.0, w1 = 0.0;
      for (int g = lane; g < RG; g += 32) {
        if (l0) w0 += __ldcg(jb.wpart + (int64_t)g * N + p0);
        if (l1) w1 += __ldcg(jb.wpart + (int64_t)g * N + p1);
      }
      w0 = tau * warp_sum(w0);
      w1 = tau * warp_sum(w1);
      double n0 = 0.0, n1 = 0.0;
      auto store = [&](double* col, int p, int64_t i, double a, double& nacc) {
        *col = a;
        if (i == j) jb.Rp[j + (int64_t)p * N] = a;
        if (i == j + 1) jb.xrow[p] = a;
        if (i >= j + 2) nacc = fma(a, a, nacc);
      };
      for (int64_t lo = b_lo; lo < r_hi; lo += RC) {
        const int rows = (int)std::min<int64_t>(RC, r_hi - lo);
        if (!keep) load_v(lo, rows);
        if (!l0) continue;
        double* ca = A + (int64_t)p0 * M + lo;
        double* cbp = A + (int64_t)p1 * M + lo;
        for (int t0 = lane; t0 < rows; t0 += 32 * HU) {
          double x[HU], y[HU];
#pragma unroll
          for (int u = 0; u < HU; ++u) {
            const bool in = t0 + 32 * u < rows;
            x[u] = in ? __ldcg(ca + t0 + 32 * u) : 0.0;
            y[u] = in && l1 ? __ldcg(cbp + t0 + 32 * u) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < HU; ++u) {
            const int t = t0 + 32 * u;
            if (t < rows) {
              store(ca + t, p0, lo + t, fma(-v[t], w0, x[u]), n0);
              if (l1) store(cbp + t, p1, lo + t, fma(-v[t], w1, y[u]), n1);
            }
          }
        }
      }
      n0 = warp_sum(n0);
      n1 = warp_sum(n1);
      if (lane == 0) {
        if (l0) jb.part[(int64_t)rg * N + p0] = n0;
        if (l1) jb.part[(int64_t)rg * N + p1] = n1;
      }
    }
    if (!grid_barrier(jb.sync, nblocks)) return;
  }
  if (lb == 0 && threadIdx.x == 0) *jb.st = HHState{0.0, N};
}

// At[l + N * i] = R[i, l] = Rp[i + N * perm[l]] for l < N, i < k: the transpose of the kept rows
__global__ void gather_rt_kernel(const double* __restrict__ Rp, int64_t N, int k,
                                 const int* __restrict__ perm, double* __restrict__ At) {
  const int64_t total = N * k;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t l = e % N, i = e / N;
    At[e] = Rp[i + N * (int64_t)perm[l]];
  }
}

// Rd[i + k * l] = R[i, l] = Rp[i + N * perm[l]] for i < k, l < N: the kept rows of R, dense,
// in pivoted column order
__global__ void gather_r_kernel(const double* __restrict__ Rp, int64_t N, int k, const int* __restrict__ perm,
                                double* __restrict__ Rd) {
  const int64_t total = N * k;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % k, l = e / k;
    Rd[e] = Rp[i + N * (int64_t)perm[l]];
  }
}

// V = I (n x n, column-major)
__global__ void eye_kernel(double* __restrict__ V, int64_t n) {
  const int64_t total = n * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x)
    V[e] = (e % n == e / n) ? 1.0 : 0.0;
}

// ---------------- one-sided Jacobi (Hestenes) with round-robin pairing -----------------
// All sweeps of one call run in a single cooperative launch with one block per SM. Round r of
// a sweep pairs the columns (a, b) of the round-robin tournament on p = ncols (+1 if odd)
// players; each warp rotates one pair at a time, and the rounds are separated by a grid
// barrier. Rotation (Rutishauser): zeta = (beta - alpha) / (2 gamma),
// t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)), c = 1/sqrt(1 + t^2), s = c t,
// [a, b] <- [c a - s b, s a + c b].
// colsq[] holds every column's squared norm (refreshed for the two columns of each
// rotation). A pair whose squared norms are both below `small2` is skipped without being
// read, and a rotation counts toward convergence only if it moves a column of squared norm
// >= `count2` by more than rounding (a rotation of a large column with a far smaller one
// changes only the smaller). The sweeps end when no such rotation is left. With
// small2 = (1e-3 delta)^2 / q and count2 = (1e-2 delta)^2 / q the columns left unsettled carry
// < 1e-4 delta^2 in total, so they change neither the kept subspace nor, except within that
// margin of the threshold, the truncation rank.
// Columns and norms written by other blocks in earlier rounds are read through L2 (ld.cg),
// never from a possibly stale L1 line. A pair's alpha and beta are read from colsq[] (the
// squared norms its last rotation, or the initial pass, summed from the stored columns), so the
// first pass over the pair only forms gamma = a.b. When V is given (vrows x ncols), every
// rotation is applied to V's columns as well, accumulating the right rotation.
constexpr int JB = 256;            // threads per block
constexpr int JU = 8;              // rows per lane per load batch
constexpr int JMAX_SWEEPS = 60;

struct JacJob {
  double* A;
  int64_t rows;
  int ncols, p;        // p: ncols, plus one if odd
  double tol, small2, count2;
  double* colsq;
  double* V;
  int64_t vrows;
};
struct JacBatch {
  JacJob j[MAX_JOBS];
  int count;
};
struct JacobiSync {                // device state of one call (zeroed before the launch)
  GridSync sync;
  int sweeps[MAX_JOBS];            // sweeps run; JMAX_SWEEPS + 1 if not converged
  unsigned rot[JMAX_SWEEPS][MAX_JOBS];  // counted rotations per sweep and matrix
};

// Several matrices share a launch: round r works on pair r of every matrix that still has one, so a
// batch of sectors costs the barriers of its largest.
__global__ void __launch_bounds__(JB) jacobi_kernel(JacBatch batch, JacobiSync* __restrict__ js) {
  const unsigned nb = gridDim.x;
  const int lane = threadIdx.x & 31;
  // pairs are dealt to blocks first (pair pr goes to block pr mod nb), so that a round's FP64
  // work spreads over every SM even when there are fewer pairs than warps
  const int gw0 = (int)(blockIdx.x + nb * (threadIdx.x >> 5));
  const int nwarps = (int)(nb * (JB / 32));
  unsigned open = (1u << batch.count) - 1u;  // matrices not yet converged
  for (int sweep = 0; sweep < JMAX_SWEEPS; ++sweep) {
    int rounds = 0;
    for (int q = 0; q < batch.count; ++q)
      if (open >> q & 1u) rounds = max(rounds, batch.j[q].p - 1);
    for (int r = 0; r < rounds; ++r) {
      int base = 0;  // pairs of the matrices before q in this round
      for (int q = 0; q < batch.count; ++q) {
        const JacJob& jb = batch.j[q];
        const int p = jb.p, npairs = p / 2;
        if (!(open >> q & 1u) || r >= p - 1) continue;
        const int ncols = jb.ncols;
        const int64_t rows = jb.rows, vrows = jb.vrows;
        const double tol = jb.tol, small2 = jb.small2, count2 = jb.count2;
        double* __restrict__ A = jb.A;
        double* __restrict__ V = jb.V;
        double* __restrict__ colsq = jb.colsq;
        // this warp's pairs among the round's: numbers gw0 + i nwarps, less the matrices before
        int first = gw0 - base % nwarps;
        if (first < 0) first += nwarps;
        base += npairs;
        for (int pr = first; pr < npairs; pr += nwarps) {
          int a, b;
          if (pr == 0) {
            a = p - 1;
            b = r;
          } else {
            a = (r + pr) % (p - 1);
            b = (r - pr + (p - 1)) % (p - 1);
          }
          if (a > b) {
            const int t = a;
            a = b;
            b = t;
          }
          if (b >= ncols) continue;  // dummy player when ncols is odd
          const double al = __ldcg(colsq + a), be = __ldcg(colsq + b);
          if (al < small2 && be < small2) continue;
          double* ca = A + (int64_t)a * rows;
          double* cb = A + (int64_t)b * rows;
          // JU rows per lane per iteration, all loads issued before the arithmetic, so that the
          // L2 latency is paid once per JU rows
          double ga = 0.0;
          for (int64_t i0 = lane; i0 < rows; i0 += 32 * JU) {
            double x[JU], y[JU];
#pragma unroll
            for (int u = 0; u < JU; ++u) {
              const int64_t i = i0 + 32 * u;
              x[u] = i < rows ? __ldcg(ca + i) : 0.0;
              y[u] = i < rows ? __ldcg(cb + i) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < JU; ++u) ga = fma(x[u], y[u], ga);
          }
          ga = warp_sum(ga);
          if (!(al > 0.0) || !(be > 0.0) || !(fabs(ga) > tol * sqrt(al) * sqrt(be))) continue;
          const double zeta = (be - al) / (2.0 * ga);
          const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
          const double cs = 1.0 / sqrt(1.0 + t * t), sn = cs * t;
          double na = 0.0, nbb = 0.0;
          for (int64_t i0 = lane; i0 < rows; i0 += 32 * JU) {
            double x[JU], y[JU];
#pragma unroll
            for (int u = 0; u < JU; ++u) {
              const int64_t i = i0 + 32 * u;
              x[u] = i < rows ? __ldcg(ca + i) : 0.0;
              y[u] = i < rows ? __ldcg(cb + i) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < JU; ++u) {
              const int64_t i = i0 + 32 * u;
              const double xa = cs * x[u] - sn * y[u], yb = sn * x[u] + cs * y[u];
              if (i < rows) {
                ca[i] = xa;
                cb[i] = yb;
              }
              na = fma(xa, xa, na);
              nbb = fma(yb, yb, nbb);
            }
          }
          if (V) {
            double* va = V + (int64_t)a * vrows;
            double* vb = V + (int64_t)b * vrows;
            for (int64_t i0 = lane; i0 < vrows; i0 += 32 * JU) {
              double x[JU], y[JU];
#pragma unroll
              for (int u = 0; u < JU; ++u) {
                const int64_t i = i0 + 32 * u;
                x[u] = i < vrows ? __ldcg(va + i) : 0.0;
                y[u] = i < vrows ? __ldcg(vb + i) : 0.0;
              }
#pragma unroll
              for (int u = 0; u < JU; ++u) {
                const int64_t i = i0 + 32 * u;
                if (i < vrows) {
                  va[i] = cs * x[u] - sn * y[u];
                  vb[i] = sn * x[u] + cs * y[u];
                }
              }
            }
          }
          na = warp_sum(na);
          nbb = warp_sum(nbb);
          if (lane == 0) {
            colsq[a] = na;
            colsq[b] = nbb;
            // the rotation counts toward convergence if it moved a column of squared norm
            // >= count2 by more than rounding: column a changes by ~|t| ||b||, column b by ~|t| ||a||
            const double move_a = al >= count2 ? fabs(t) * sqrt(be / al) : 0.0;
            const double move_b = be >= count2 ? fabs(t) * sqrt(al / be) : 0.0;
            if (fmax(move_a, move_b) > 4.0 * 2.220446049250313e-16) atomicAdd(&js->rot[sweep][q], 1u);
          }
        }
      }
      if (!grid_barrier(&js->sync, nb)) return;
    }
    // after the sweep's last barrier every block reads the same final counts
    for (int q = 0; q < batch.count; ++q)
      if ((open >> q & 1u) && *(volatile unsigned*)&js->rot[sweep][q] == 0) {
        open &= ~(1u << q);
        if (blockIdx.x == 0 && threadIdx.x == 0) js->sweeps[q] = sweep + 1;
      }
    if (!open) return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0)
    for (int q = 0; q < batch.count; ++q)
      if (open >> q & 1u) js->sweeps[q] = JMAX_SWEEPS + 1;
}

__global__ void colsq_init_kernel(const double* __restrict__ A, int64_t rows, int ncols,
                                  double* __restrict__ colsq) {
  const int gw = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (gw >= ncols) return;
  const double* col = A + (int64_t)gw * rows;
  double acc = 0.0;
  for (int64_t i = lane; i < rows; i += 32) acc = fma(col[i], col[i], acc);
  acc = warp_sum(acc);
  if (lane == 0) colsq[gw] = acc;
}


// norms[c] = ||A[:, c]||_2, one warp per column
__global__ void colnorm_kernel(const double* __restrict__ A, int64_t rows, int ncols,
                               double* __restrict__ norms) {
  const int gw = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (gw >= ncols) return;
  const double* col = A + (int64_t)gw * rows;
  double acc = 0.0;
  for (int64_t i = lane; i < rows; i += 32) acc = fma(col[i], col[i], acc);
  acc = warp_sum(acc);
  if (lane == 0) norms[gw] = sqrt(acc);
}

// out[:, q] = in[:, perm[q]] * (scale ? 1/norms[perm[q]] : 1), q < r
__global__ void gather_cols_kernel(const double* __restrict__ in, int64_t rows,
                                   const int* __restrict__ perm, int r,
                                   const double* __restrict__ norms, double* __restrict__ out) {
  const int64_t total = rows * r;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % rows;
    const int q = (int)(e / rows);
    const int src = perm[q];
    double val = in[i + (int64_t)src * rows];
    if (norms) {
      const double nr = norms[src];
      val = nr > 0.0 ? val / nr : 0.0;
    }
    out[e] = val;
  }
}

// out[perm[i] + rows q] = in[i + rows q] (rows x ncols, column-major)
__global__ void scatter_rows_kernel(const double* __restrict__ in, int64_t rows, int ncols,
                                    const int* __restrict__ perm, double* __restrict__ out) {
  const int64_t total = rows * ncols;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e % rows, q = e / rows;
    out[perm[i] + q * rows] = in[e];
  }
}

__global__ void cast_f32_kernel(const double* __restrict__ in, int64_t n, float* __restrict__ out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (float)in[e];
}

__global__ void widen_f32_kernel(const float* __restrict__ in, int64_t n, double* __restrict__ out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (double)in[e];
}

// ---------------- FP64 SIMT GEMM (column-major) -------------------------------------
// C[gm rc + gn cc] = alpha sum_k op(A)[gm, k] op(B)[k, gn] + beta C, blocks of BM x BN outputs (TY x 256 / TY
// threads of TM x TN each), K in chunks of 16, blockIdx.z taking its slice of K. With more than one slice the
// sums go to part (slice, gn M + gm) and dgemm_reduce_kernel adds the slices in order. The FP64 pipe takes 16 clocks per
// warp FMA, so any tile keeps it busy; what costs is padding (outputs computed for rows past M) and idle SMs, and
// dgemm() picks the tile and the slices against those.
template <int TY, int TM, int TN>
__global__ void __launch_bounds__(256)
    dgemm_kernel(bool tA, bool tB, int64_t M, int64_t N, int64_t K, int64_t kslice, double alpha,
                 const double* __restrict__ A, int64_t lda, const double* __restrict__ B, int64_t ldb, double beta,
                 double* __restrict__ C, int64_t rc, int64_t cc, double* __restrict__ part) {
  constexpr int TX = 256 / TY, BM = TY * TM, BN = TX * TN, BK = 16;
  __shared__ double As[BK][BM + 1];
  __shared__ double Bs[BK][BN + 1];
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  const int64_t m0 = (int64_t)blockIdx.y * BM, n0 = (int64_t)blockIdx.x * BN;
  const int64_t k_lo = blockIdx.z * kslice, k_hi = std::min<int64_t>(K, k_lo + kslice);
  double acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;
  for (int64_t k0 = k_lo; k0 < k_hi; k0 += BK) {
#pragma unroll
    for (int e0 = 0; e0 < (BM * BK + 255) / 256; ++e0) {
      const int e = e0 * 256 + threadIdx.x;
      if (BM * BK % 256 != 0 && e >= BM * BK) break;
      int mm, kk;
      if (tA) { kk = e % BK; mm = e / BK; } else { mm = e % BM; kk = e / BM; }
      const int64_t gm = m0 + mm, gk = k0 + kk;
      double val = 0.0;
      if (gm < M && gk < k_hi) val = tA ? A[gk + gm * lda] : A[gm + gk * lda];
      As[kk][mm] = val;
    }
#pragma unroll
    for (int e0 = 0; e0 < BN * BK / 256; ++e0) {
      const int e = e0 * 256 + threadIdx.x;
      int nn, kk;
      if (tB) { nn = e % BN; kk = e / BN; } else { kk = e % BK; nn = e / BK; }
      const int64_t gn = n0 + nn, gk = k0 + kk;
      double val = 0.0;
      if (gn < N && gk < k_hi) val = tB ? B[gn + gk * ldb] : B[gk + gn * ldb];
      Bs[kk][nn] = val;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      double a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty * TM + i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + TX * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < TN; ++j) {
    const int64_t gn = n0 + tx + TX * j;
    if (gn >= N) continue;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int64_t gm = m0 + ty * TM + i;
      if (gm >= M) continue;
      if (part) {
        part[(int64_t)blockIdx.z * M * N + gn * M + gm] = acc[i][j];
      } else {
        double* cp = C + gm * rc + gn * cc;
        *cp = alpha * acc[i][j] + (beta == 0.0 ? 0.0 : beta * *cp);
      }
    }
  }
}

__global__ void __launch_bounds__(256) dgemm_reduce_kernel(const double* __restrict__ part, int slices, int64_t M, int64_t N,
                                                           double alpha, double beta, double* __restrict__ C, int64_t rc, int64_t cc) {
  const int64_t total = M * N;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int z = 0; z < slices; ++z) acc += part[z * total + e];
    double* cp = C + e % M * rc + e / M * cc;
    *cp = alpha * acc + (beta == 0.0 ? 0.0 : beta * *cp);
  }
}

// Stream-ordered scratch.
struct Buf {
  double* p = nullptr;
  cudaStream_t s = nullptr;
  Buf() = default;
  Buf(const Buf&) = delete;
  Buf& operator=(const Buf&) = delete;
  Buf(Buf&& o) noexcept : p(o.p), s(o.s) { o.p = nullptr; }
  Buf& operator=(Buf&& o) noexcept {
    std::swap(p, o.p);
    std::swap(s, o.s);
    return *this;
  }
  ~Buf() { free(); }
  void free() {
    if (p) cudaFreeAsync(p, s);
    p = nullptr;
  }
  pttk_status alloc(size_t elems, cudaStream_t st) {
    free();
    s = st;
    if (elems == 0) elems = 1;
    const cudaError_t e = ws_malloc(&p, elems * sizeof(double), st);
    if (e != cudaSuccess) {
      p = nullptr;
      cudaGetLastError();
      return set_error(PTTK_ENOMEM, "device allocation failed in TT-SVD");
    }
    return PTTK_OK;
  }
  pttk_status alloc_ints(size_t count, cudaStream_t st) { return alloc((count + 1) / 2, st); }
  int* ints() const { return reinterpret_cast<int*>(p); }
};

unsigned grid1d(int64_t work, int threads, int cap_per_sm = 8) {
  const int64_t b = (work + threads - 1) / threads;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)sm_count() * cap_per_sm));
}

// Blocks of a cooperative kernel that are resident together.
template <typename K>
pttk_status coop_capacity(K kernel, int threads, size_t smem, int* blocks) {
  int per_sm = 0;
  PTTK_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
  if (per_sm < 1) return set_error(PTTK_ECUDA, "cooperative kernel cannot be resident");
  *blocks = per_sm * sm_count();
  return PTTK_OK;
}

// Pivoted Householder QR of A (M x N, M >= N, overwritten), stopped once ||R22||_F^2 <= stop2
// (at least one step is taken). On return perm[0..N) holds the column order, Rp the rows
// 0..k-1 of R by physical column (N x N, zeroed here), k the number of rows kept and tail2
// ||R22||_F^2 at the stop. A batch runs in one launch; synchronises `s`.
struct Qr {
  double* A;
  int64_t M;
  int N;
  double stop2;
  double* Rp;
  int* perm;
  int k = 0;
  double tail2 = 0.0;
};
pttk_status householder_batch(std::vector<Qr>& qr, cudaStream_t s) {
  PTTK_PROF("householder", s);
  const int count = (int)qr.size();
  int nmax = 1;
  for (const Qr& q : qr) nmax = std::max(nmax, q.N);
  const size_t smem = (sizeof(unsigned) + sizeof(int)) * (((size_t)nmax + 31) / 32);
  double total = 0.0;
  for (const Qr& q : qr) total += (double)q.M * q.N;
  auto kfn = total >= 8e6 ? hh_kernel<3, 4096> : hh_kernel<2, 1024>;
  if (smem > 8 * 1024)
    PTTK_CUDA(allow_smem((const void*)kfn));
  int cap = 0;
  PTTK_TRY(coop_capacity(kfn, 256, smem, &cap));
  QrBatch b{};
  b.count = count;
  int next = 0;
  size_t words = 0;
  for (int i = 0; i < count; ++i) {
    QrJob& j = b.j[i];
    j.A = qr[i].A;
    j.M = qr[i].M;
    j.N = qr[i].N;
    j.stop2 = qr[i].stop2;
    j.Rp = qr[i].Rp;
    j.perm = qr[i].perm;
    const int share = std::max(1, (int)((double)(cap - count) * ((double)j.M * j.N / total)));
    // a column set for each QC columns, and row groups of at least 64 rows; one group more, with fewer sets, where the sets
    // leave over a fifth of the share idle (3696 columns: 231 sets in a share of 456)
    j.cn = std::max(1, std::min(share, (j.N + QC - 1) / QC));
    j.rg = share / j.cn;
    if (5 * j.rg * j.cn < 4 * share) j.cn = share / ++j.rg;
    if (j.rg > j.M / 64) {
      j.rg = (int)std::max<int64_t>(1, j.M / 64);
      j.cn = std::max(1, std::min(share / j.rg, (j.N + QC - 1) / QC));
    }
    j.block0 = next;
    next += j.cn * j.rg;
    words += ((size_t)2 * j.rg + 1) * j.N;
  }
  Buf work, sync;
  PTTK_TRY(work.alloc(words, s));
  const size_t per = sizeof(GridSync) + 128;  // the barrier, then the result
  PTTK_TRY(sync.alloc(per * count / sizeof(double), s));
  PTTK_CUDA(cudaMemsetAsync(sync.p, 0, per * count, s));
  size_t off = 0;
  for (int i = 0; i < count; ++i) {
    QrJob& j = b.j[i];
    j.part = work.p + off;
    j.wpart = j.part + (size_t)j.rg * j.N;
    j.xrow = j.wpart + (size_t)j.rg * j.N;
    off += ((size_t)2 * j.rg + 1) * j.N;
    char* base = reinterpret_cast<char*>(sync.p) + per * i;
    j.sync = reinterpret_cast<GridSync*>(base);
    j.st = reinterpret_cast<HHState*>(base + sizeof(GridSync));
    PTTK_CUDA(cudaMemsetAsync(j.Rp, 0, sizeof(double) * (size_t)j.N * j.N, s));
  }
  void* args[] = {&b};
  PTTK_CUDA(cudaLaunchCooperativeKernel((const void*)kfn, dim3((unsigned)next), dim3(256), args, smem, s));
  pttk::count_launch();
  std::vector<char> host(per * count);
  PTTK_CUDA(cudaMemcpyAsync(host.data(), sync.p, per * count, cudaMemcpyDeviceToHost, s));
  PTTK_CUDA(cudaStreamSynchronize(s));
  for (int i = 0; i < count; ++i) {
    GridSync g;
    HHState h;
    memcpy(&g, host.data() + per * i, sizeof g);
    memcpy(&h, host.data() + per * i + sizeof(GridSync), sizeof h);
    if (g.err) return set_error(PTTK_ETIMEOUT, "pivoted QR: a grid barrier timed out");
    qr[i].k = h.k;
    qr[i].tail2 = h.tail2;
  }
  return PTTK_OK;
}

// One-sided Jacobi on the columns of A (rows x ncols), all sweeps of a batch in one cooperative launch;
// synchronises `s` once to read the outcome. With V (vrows x ncols), every rotation is also
// applied to V's columns. Columns of norm below `small` are not rotated against each other.
struct Jac {
  double* A;
  int64_t rows;
  int ncols;
  double small = 0.0;
  double* V = nullptr;
  int64_t vrows = 0;
};
pttk_status jacobi_batch(const std::vector<Jac>& all, cudaStream_t s) {
  std::vector<Jac> jobs;
  int64_t cols = 0;
  int pairs = 0;
  for (const Jac& j : all)
    if (j.ncols >= 2) {
      jobs.push_back(j);
      cols += j.ncols;
      pairs += (j.ncols + 1) / 2;
    }
  if (jobs.empty()) return PTTK_OK;
  Buf colsq, state;
  PTTK_TRY(colsq.alloc(cols, s));
  PTTK_TRY(state.alloc((sizeof(JacobiSync) + sizeof(double) - 1) / sizeof(double), s));
  static_assert(alignof(JacobiSync) <= 256, "device allocation alignment");
  JacobiSync* js = reinterpret_cast<JacobiSync*>(state.p);
  PTTK_CUDA(cudaMemsetAsync(js, 0, sizeof(JacobiSync), s));
  JacBatch b{};
  b.count = (int)jobs.size();
  double* cs = colsq.p;
  for (int i = 0; i < b.count; ++i) {
    const Jac& j = jobs[i];
    colsq_init_kernel<<<(unsigned)(((int64_t)j.ncols * 32 + 255) / 256), 256, 0, s>>>(j.A, j.rows, j.ncols, cs); pttk::count_launch();
    const double small2 = j.small * j.small;
    // A pair counts as orthogonal once |a.b| <= sqrt(rows) eps ||a|| ||b||: the typical rounding
    // level of a computed dot product. The singular subspaces are then accurate to that level,
    // which the 1e-12 parity of K~ needs (a looser rows * eps stops ~20x earlier in accuracy).
    const double tol = sqrt((double)std::max<int64_t>(j.rows, 16)) * 2.220446049250313e-16;
    b.j[i] = JacJob{j.A, j.rows, j.ncols, j.ncols + (j.ncols & 1), tol, small2, 100.0 * small2, cs, j.V, j.vrows};
    cs += j.ncols;
  }
  {
    PTTK_PROF("jacobi", s);
    int cap = 0;
    PTTK_TRY(coop_capacity(jacobi_kernel, JB, 0, &cap));
    // one block per SM (fewer when there are fewer pairs); each block takes up to 8 pairs of a
    // round at a time, pairs dealt round-robin over the blocks
    const unsigned grid = (unsigned)std::max(1, std::min({pairs, sm_count(), cap}));
    void* args[] = {&b, &js};
    PTTK_CUDA(cudaLaunchCooperativeKernel((const void*)jacobi_kernel, dim3(grid), dim3(JB), args, 0, s));
    pttk::count_launch();
  }
  JacobiSync h{};
  PTTK_CUDA(cudaMemcpyAsync(&h, js, sizeof(JacobiSync), cudaMemcpyDeviceToHost, s));
  PTTK_CUDA(cudaStreamSynchronize(s));
  if (kDebugLog)
    for (int i = 0; i < b.count; ++i)
      fprintf(stderr, "pttk: jacobi %lld x %d sweeps %d\n", (long long)b.j[i].rows, b.j[i].ncols, h.sweeps[i]);
  if (h.sync.err) return set_error(PTTK_ETIMEOUT, "one-sided Jacobi: a grid barrier timed out");
  for (int i = 0; i < b.count; ++i)
    if (h.sweeps[i] > JMAX_SWEEPS) return set_error(PTTK_ECUDA, "one-sided Jacobi SVD did not converge in 60 sweeps");
  return PTTK_OK;
}

// Sorted order of sigma (descending) and the truncation rank for threshold delta.
// `extra2` is a squared norm already discarded (the R22 of a truncated QR), counted in every tail.
int truncation(const std::vector<double>& sigma, double delta, std::vector<int>& perm, double extra2 = 0.0) {
  perm.resize(sigma.size());
  std::iota(perm.begin(), perm.end(), 0);
  std::stable_sort(perm.begin(), perm.end(), [&](int x, int y) { return sigma[x] > sigma[y]; });
  const int m = (int)sigma.size();
  std::vector<double> tail(m + 1, 0.0);  // tail[r] = extra2 + sum_{i >= r} sigma_(i)^2
  tail[m] = extra2;
  for (int i = m - 1; i >= 0; --i) tail[i] = tail[i + 1] + sigma[perm[i]] * sigma[perm[i]];
  for (int r = 1; r <= m; ++r)
    if (sqrt(tail[r]) <= delta) return r;
  return m;
}

}  // namespace

// Tile: up to M = 256 the one of BM in {4, 8, 12, 16, 24, 32, 40, 48, 64} with the least padding of M (the larger of
// equals), 64 above (padding no longer counts, and the grid's y stays as short as it was); the product is taken
// transposed where N is the smaller side below 64, so that the padding fits it (Q y over N = 12,000 points took 13 ms
// in 64 x 64 tiles of one column). Slices of K, of at least 64: where the tiles are fewer than two per SM.
// All products of the marginal likelihood at N = 12,000: 14.4 -> 0.36 ms; of a 20^5 TT-SVD: 2.7 -> 0.62 ms; of a 12^8
// one: 32.6 -> 14.2 ms.
void dgemm(bool tA, bool tB, int64_t M, int64_t N, int64_t K, double alpha, const double* A,
           int64_t lda, const double* B, int64_t ldb, double beta, double* C, int64_t ldc,
           cudaStream_t s) {
  if (M <= 0 || N <= 0) return;
  PTTK_PROF("dgemm", s);
  int64_t rc = 1, cc = ldc;
  if (N < M && N < 64) {
    std::swap(A, B);
    std::swap(lda, ldb);
    std::swap(M, N);
    std::swap(rc, cc);
    const bool t = tA;
    tA = !tB;
    tB = !t;
  }
  int bm = M > 256 ? 64 : 4;
  for (int t : {8, 12, 16, 24, 32, 40, 48, 64})
    if (t > bm && (M + t - 1) / t * t <= (M + bm - 1) / bm * bm) bm = t;
  const int bn = bm == 64 ? 64 : 128;
  const int64_t gx = (N + bn - 1) / bn, gy = (M + bm - 1) / bm;
  int64_t slices = std::max<int64_t>(1, std::min<int64_t>((int64_t)sm_count() * 2 / std::max<int64_t>(gx * gy, 1), K / 64));
  slices = std::min<int64_t>(slices, 1024);
  int64_t kslice = std::max<int64_t>(K, 1);
  double* part = nullptr;
  if (slices > 1) {
    kslice = ((K + slices - 1) / slices + 15) / 16 * 16;
    slices = (K + kslice - 1) / kslice;
    if (slices < 2 || ws_malloc(&part, sizeof(double) * (size_t)slices * M * N, s) != cudaSuccess) {
      cudaGetLastError();
      part = nullptr;
      slices = 1;
      kslice = std::max<int64_t>(K, 1);
    }
  }
  const dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)slices);
  auto run = [&](auto kfn) {
    kfn<<<grid, 256, 0, s>>>(tA, tB, M, N, K, kslice, alpha, A, lda, B, ldb, beta, C, rc, cc, part);
    pttk::count_launch();
  };
  switch (bm) {
    case 4: run(dgemm_kernel<4, 1, 2>); break;
    case 8: run(dgemm_kernel<4, 2, 2>); break;
    case 12: run(dgemm_kernel<4, 3, 2>); break;
    case 16: run(dgemm_kernel<4, 4, 2>); break;
    case 24: run(dgemm_kernel<8, 3, 4>); break;
    case 32: run(dgemm_kernel<8, 4, 4>); break;
    case 40: run(dgemm_kernel<8, 5, 4>); break;
    case 48: run(dgemm_kernel<8, 6, 4>); break;
    default: run(dgemm_kernel<16, 4, 4>); break;
  }
  if (part) {
    dgemm_reduce_kernel<<<grid1d(M * N, 256), 256, 0, s>>>(part, (int)slices, M, N, alpha, beta, C, rc, cc); pttk::count_launch();
    cudaFreeAsync(part, s);
  }
}

// Wall-clock stage timing of the TT-SVD, printed to stderr in a PTTK_DEBUG build (it
// synchronises the stream at every mark, so release builds compile it out).
struct StageClock {
  bool on;
  cudaStream_t s;
  std::chrono::steady_clock::time_point t0;
  explicit StageClock(cudaStream_t st) : on(kDebugLog), s(st) { reset(); }
  void reset() {
    if (!on) return;
    cudaStreamSynchronize(s);
    t0 = std::chrono::steady_clock::now();
  }
  void mark(int k, const char* what) {
    if (!on) return;
    cudaStreamSynchronize(s);
    const auto t1 = std::chrono::steady_clock::now();
    fprintf(stderr, "pttk: tt-svd step %d %-10s %9.3f ms\n", k + 1, what,
            std::chrono::duration<double, std::milli>(t1 - t0).count());
    t0 = t1;
  }
};

// One matrix X (m x c, column-major, not modified) on its way to a basis of its leading left singular
// subspace: an unfolding, or the block of one parity sector of it.
struct SvdPart {
  const double* X = nullptr;
  int64_t m = 0, c = 0;
  bool wide() const { return c >= m; }
  int64_t q() const { return wide() ? m : c; }    // columns of the QR input
  int64_t Mqr() const { return wide() ? c : m; }  // rows of the QR input
  Buf qrin, R, A, perm;
  int kq = 0;
  double tail2 = 0.0;
  std::vector<double> sigma;  // singular values, in the order of A's columns
  int r = 0;                  // leading ones to keep
  Buf core;                   // m x r, unit columns in decreasing singular value
};

// Cuts the parts' kept rows back to where the pivoted QR of all of them together reaches ||R22||^2 <= stop2
// (see svd_factor); A = R1^T keeps its leading columns.
static pttk_status cut_parts(std::vector<SvdPart>& parts, double stop2, cudaStream_t s) {
  const size_t np = parts.size();
  std::vector<std::vector<double>> diag(np), row(np);  // |R_jj|, ||R[j, :]||
  std::vector<Buf> norms(np);
  for (size_t i = 0; i < np; ++i) {
    SvdPart& pt = parts[i];
    if (pt.kq == 0) continue;
    const int64_t q = pt.q();
    diag[i].resize(pt.kq);
    row[i].resize(pt.kq);
    PTTK_TRY(norms[i].alloc(pt.kq, s));
    colnorm_kernel<<<(unsigned)(((int64_t)pt.kq * 32 + 255) / 256), 256, 0, s>>>(pt.A.p, q, pt.kq, norms[i].p); pttk::count_launch();
    PTTK_CUDA(cudaMemcpyAsync(row[i].data(), norms[i].p, sizeof(double) * pt.kq, cudaMemcpyDeviceToHost, s));
    PTTK_CUDA(cudaMemcpy2DAsync(diag[i].data(), sizeof(double), pt.A.p, sizeof(double) * (q + 1), sizeof(double), pt.kq,
                                cudaMemcpyDeviceToHost, s));
  }
  PTTK_CUDA(cudaStreamSynchronize(s));
  // left[i][j]: the square of part i's block after j steps, summed from its end
  std::vector<std::vector<double>> left(np);
  std::vector<int> at(np, 0);
  for (size_t i = 0; i < np; ++i) {
    left[i].assign(parts[i].kq + 1, parts[i].tail2);
    for (int j = parts[i].kq - 1; j >= 0; --j) left[i][j] = left[i][j + 1] + row[i][j] * row[i][j];
  }
  while (true) {
    double sum = 0.0;
    for (size_t i = 0; i < np; ++i) sum += left[i][at[i]];
    if (sum <= stop2) break;
    int next = -1;
    for (size_t i = 0; i < np; ++i)
      if (at[i] < parts[i].kq && (next < 0 || fabs(diag[i][at[i]]) > fabs(diag[next][at[next]]))) next = (int)i;
    if (next < 0) break;
    ++at[next];
  }
  for (size_t i = 0; i < np; ++i) {
    const int k = std::max(at[i], std::min(1, parts[i].kq));
    parts[i].kq = k;
    parts[i].tail2 = left[i][k];
  }
  return PTTK_OK;
}

// Factors the parts: R1^T V = U' Sigma of the kept rows R1 of the pivoted QR (A holds U' Sigma), with the
// singular values. delta and stop_frac: the pivoted QRs stop once their discarded blocks together have
// ||R22||_F <= stop_frac delta.
//
// Several parts stop where the pivoted QR of the whole unfolding would. That QR takes the part with the
// largest trailing column at each step and leaves the others alone, so its steps are the parts' own, merged by
// decreasing |R_jj|. Each part factors until its block is a sixteenth of its share (in squares), and the host cuts
// the parts back to the step of the merged order at which the blocks together are small enough: the kept rows,
// and with them the ranks of unfoldings whose tail lies within stop_frac^2 of the threshold, are
// those of one QR.
static pttk_status svd_factor(std::vector<SvdPart>& parts, double delta, double stop_frac, StageClock& clk, int k,
                              cudaStream_t s) {
  const int np = (int)parts.size();
  clk.reset();
  // QR input: wide -> W = X^T (c x m), tall -> a copy of X (m x c). The pivoted QR makes
  // the triangular factor graded, so one-sided Jacobi on its transpose converges in a few
  // sweeps, and stops once the remaining block is negligible next to delta.
  std::vector<Qr> qr;
  // rows of R kept: the QR stops once the discarded block has ||R22||_F <= stop_frac delta
  // (0.03 for the TT-SVD). The tails below count ||R22||^2, so the error bound of the
  // truncation holds as it is; only a tail within stop_frac^2 delta^2 of the threshold could
  // give a rank one higher than the exact singular values would. The discarded block also
  // moves the kept subspace by about stop_frac delta against the exact SVD's
  const double stop = stop_frac * delta;
  for (SvdPart& pt : parts) {
    const int64_t q = pt.q(), Mqr = pt.Mqr();
    if (clk.on) fprintf(stderr, "pttk: tt-svd step %d m %lld c %lld %s\n", k + 1, (long long)pt.m, (long long)pt.c, pt.wide() ? "wide" : "tall");
    PTTK_TRY(pt.perm.alloc_ints(q, s));
    PTTK_TRY(pt.qrin.alloc(Mqr * q, s));
    if (pt.wide()) {
      dim3 tg((unsigned)((pt.c + 31) / 32), (unsigned)((pt.m + 31) / 32));
      transpose_kernel<<<tg, dim3(32, 8), 0, s>>>(pt.X, pt.m, pt.c, nullptr, pt.qrin.p); pttk::count_launch();
    } else {
      PTTK_CUDA(cudaMemcpyAsync(pt.qrin.p, pt.X, sizeof(double) * pt.m * pt.c, cudaMemcpyDeviceToDevice, s));
    }
    PTTK_TRY(pt.R.alloc(q * q, s));
    qr.push_back(Qr{pt.qrin.p, Mqr, (int)q, np == 1 ? stop * stop : stop * stop / (16.0 * np), pt.R.p, pt.perm.ints()});
  }
  clk.mark(k, "layout");
  PTTK_TRY(householder_batch(qr, s));
  clk.mark(k, "qr");
  // one-sided Jacobi on A = R1^T (q x kq), R1 = the kept rows of R in pivoted column order: R1^T V = U'
  // Sigma, so R1 = V Sigma U'^T and the right singular vectors of R1 (= of the pivoted QR input, up to
  // the discarded R22) are the normalised columns of the rotated R1^T; columns below (stop_frac / 30)
  // delta / sqrt(kq), kq over all parts, together carry < (stop_frac / 30)^2 delta^2, and pairs of them are skipped.
  // Where R1^T has at least 2.5 times as many rows as columns: a second pivoted QR, R1^T P2 = Q2 R2, and
  // the Jacobi on R2 (kq x kq), whose columns have the Gram matrix of R1^T P2's and so take the same
  // rotations, accumulated in V; the rotated R1^T is then R1^T (P2 V), one DGEMM. Each rotation touches
  // 2 kq rows (R2 and V) instead of q. The second QR and the fixed cost of a Jacobi round (L2 round
  // trips, grid barrier) eat the gain below that ratio.
  struct Second {
    SvdPart* pt;
    Buf A0, R, perm, Rd, V, PV;
  };
  std::vector<Second> second;
  std::vector<Qr> qr2;
  std::vector<Jac> jac;
  for (int i = 0; i < np; ++i) {
    SvdPart& pt = parts[i];
    const int64_t q = pt.q();
    pt.kq = qr[i].k;
    pt.tail2 = qr[i].tail2;
    pt.qrin.free();
    PTTK_TRY(pt.A.alloc(q * pt.kq, s));
    gather_rt_kernel<<<grid1d(q * pt.kq, 256), 256, 0, s>>>(pt.R.p, q, pt.kq, pt.perm.ints(), pt.A.p); pttk::count_launch();
  }
  if (np > 1) PTTK_TRY(cut_parts(parts, stop * stop, s));
  double kq_all = 0.0;
  for (const SvdPart& pt : parts) kq_all += pt.kq;
  const double skip = (stop_frac / 30.0) * delta / sqrt(kq_all);
  for (SvdPart& pt : parts) {
    const int64_t q = pt.q();
    if (clk.on) fprintf(stderr, "pttk: tt-svd step %d kept %d of %lld rows of R, ||R22|| %.3e\n", k + 1, pt.kq, (long long)q, sqrt(pt.tail2));
    if (2 * q >= 5 * (int64_t)pt.kq && pt.kq >= 2) second.push_back(Second{&pt});
    else jac.push_back(Jac{pt.A.p, q, pt.kq, skip});
  }
  for (Second& sc : second) {
    const int64_t q = sc.pt->q(), kq = sc.pt->kq;
    PTTK_TRY(sc.A0.alloc(q * kq, s));
    PTTK_CUDA(cudaMemcpyAsync(sc.A0.p, sc.pt->A.p, sizeof(double) * q * kq, cudaMemcpyDeviceToDevice, s));
    PTTK_TRY(sc.perm.alloc_ints(kq, s));
    PTTK_TRY(sc.R.alloc(kq * kq, s));
    qr2.push_back(Qr{sc.pt->A.p, q, (int)kq, -1.0, sc.R.p, sc.perm.ints()});  // stop2 < 0: every column is factored
  }
  if (!qr2.empty()) PTTK_TRY(householder_batch(qr2, s));
  for (size_t i = 0; i < second.size(); ++i) {
    Second& sc = second[i];
    const int64_t kq = sc.pt->kq, k2 = qr2[i].k;
    PTTK_TRY(sc.Rd.alloc(k2 * kq, s));
    gather_r_kernel<<<grid1d(k2 * kq, 256), 256, 0, s>>>(sc.R.p, kq, (int)k2, sc.perm.ints(), sc.Rd.p); pttk::count_launch();
    PTTK_TRY(sc.V.alloc(kq * kq, s));
    PTTK_TRY(sc.PV.alloc(kq * kq, s));
    eye_kernel<<<grid1d(kq * kq, 256), 256, 0, s>>>(sc.V.p, kq); pttk::count_launch();
    jac.push_back(Jac{sc.Rd.p, k2, (int)kq, skip, sc.V.p, kq});
  }
  PTTK_TRY(jacobi_batch(jac, s));
  for (Second& sc : second) {
    const int64_t q = sc.pt->q(), kq = sc.pt->kq;
    // P2 V: row perm2[l] of the result is row l of V
    scatter_rows_kernel<<<grid1d(kq * kq, 256), 256, 0, s>>>(sc.V.p, kq, (int)kq, sc.perm.ints(), sc.PV.p); pttk::count_launch();
    dgemm(false, false, q, kq, kq, 1.0, sc.A0.p, q, sc.PV.p, kq, 0.0, sc.pt->A.p, q, s);
  }
  PTTK_CUDA(cudaGetLastError());
  clk.mark(k, "jacobi");
  std::vector<Buf> norms(np);
  for (int i = 0; i < np; ++i) {
    SvdPart& pt = parts[i];
    PTTK_TRY(norms[i].alloc(pt.kq, s));
    colnorm_kernel<<<(unsigned)(((int64_t)pt.kq * 32 + 255) / 256), 256, 0, s>>>(pt.A.p, pt.q(), pt.kq, norms[i].p); pttk::count_launch();
    pt.sigma.resize(pt.kq);
    PTTK_CUDA(cudaMemcpyAsync(pt.sigma.data(), norms[i].p, sizeof(double) * pt.kq, cudaMemcpyDeviceToHost, s));
  }
  PTTK_CUDA(cudaStreamSynchronize(s));
  return PTTK_OK;
}

// The kept left singular vectors of every part (its r set), in `core`.
static pttk_status svd_finish(std::vector<SvdPart>& parts, StageClock& clk, int k, cudaStream_t s) {
  const int np = (int)parts.size();
  struct Work {
    Buf order, norms, Y, U, Yt, bn;
    std::vector<int> perm;
    std::vector<double> bnh;
    double* basis = nullptr;
  };
  std::vector<Work> w(np);
  std::vector<Jac> jac;
  for (int i = 0; i < np; ++i) {
    SvdPart& pt = parts[i];
    if (pt.r == 0) continue;
    const int64_t q = pt.q(), r = pt.r;
    truncation(pt.sigma, 0.0, w[i].perm);  // decreasing order
    PTTK_TRY(w[i].order.alloc_ints(std::max<int64_t>(pt.kq, pt.r), s));
    PTTK_CUDA(cudaMemcpyAsync(w[i].order.ints(), w[i].perm.data(), sizeof(int) * pt.kq, cudaMemcpyHostToDevice, s));
    PTTK_TRY(w[i].norms.alloc(pt.kq, s));
    PTTK_CUDA(cudaMemcpyAsync(w[i].norms.p, pt.sigma.data(), sizeof(double) * pt.kq, cudaMemcpyHostToDevice, s));
    // top-r right singular vectors (unit columns), in the pivoted order
    PTTK_TRY(w[i].U.alloc(q * r, s));
    PTTK_TRY(w[i].Y.alloc(q * r, s));
    gather_cols_kernel<<<grid1d(q * r, 256), 256, 0, s>>>(pt.A.p, q, w[i].order.ints(), pt.r, w[i].norms.p, w[i].Y.p); pttk::count_launch();
    // back to the original order: row perm[l] of the result is row l of Y
    scatter_rows_kernel<<<grid1d(q * r, 256), 256, 0, s>>>(w[i].Y.p, q, pt.r, pt.perm.ints(), w[i].U.p); pttk::count_launch();
    w[i].basis = w[i].U.p;  // m x r (wide): left singular vectors of X
    if (!pt.wide()) {
      // tall: U holds the top right singular vectors of X (c x r); Y = X U spans the top-r
      // left singular subspace
      PTTK_TRY(w[i].Yt.alloc(pt.m * r, s));
      dgemm(false, false, pt.m, r, pt.c, 1.0, pt.X, pt.m, w[i].U.p, pt.c, 0.0, w[i].Yt.p, pt.m, s);
      w[i].basis = w[i].Yt.p;
    }
    jac.push_back(Jac{w[i].basis, pt.m, pt.r});
  }
  // make each basis orthonormal to working precision: its columns are orthogonal up
  // to ~eps ||X|| / sigma_i, so one-sided Jacobi needs one or two sweeps
  clk.mark(k, "basis");
  PTTK_TRY(jacobi_batch(jac, s));
  clk.mark(k, "reorth");
  for (int i = 0; i < np; ++i) {
    SvdPart& pt = parts[i];
    if (pt.r == 0) continue;
    PTTK_TRY(w[i].bn.alloc(pt.r, s));
    colnorm_kernel<<<(unsigned)(((int64_t)pt.r * 32 + 255) / 256), 256, 0, s>>>(w[i].basis, pt.m, pt.r, w[i].bn.p); pttk::count_launch();
    w[i].bnh.resize(pt.r);
    PTTK_CUDA(cudaMemcpyAsync(w[i].bnh.data(), w[i].bn.p, sizeof(double) * pt.r, cudaMemcpyDeviceToHost, s));
  }
  PTTK_CUDA(cudaStreamSynchronize(s));
  for (int i = 0; i < np; ++i) {
    SvdPart& pt = parts[i];
    if (pt.r == 0) continue;
    truncation(w[i].bnh, 0.0, w[i].perm);
    PTTK_CUDA(cudaMemcpyAsync(w[i].order.ints(), w[i].perm.data(), sizeof(int) * pt.r, cudaMemcpyHostToDevice, s));
    PTTK_TRY(pt.core.alloc(pt.m * pt.r, s));
    gather_cols_kernel<<<grid1d(pt.m * pt.r, 256), 256, 0, s>>>(w[i].basis, pt.m, w[i].order.ints(), pt.r, w[i].bn.p, pt.core.p); pttk::count_launch();
  }
  PTTK_CUDA(cudaStreamSynchronize(s));
  return PTTK_OK;
}

// Orthonormal basis (m x r, unit columns in decreasing singular value, column-major, into
// `core`) of the top-r left singular subspace of X (m x c, column-major, not modified), r the
// smallest rank >= 1 whose discarded tail sqrt(sum_{i>r} sigma_i^2) is <= delta; delta = 0
// keeps every direction X has (an orthonormal basis of its range). stop_frac: the pivoted QR
// stops once the discarded block has ||R22||_F <= stop_frac delta (see svd_factor).
static pttk_status svd_basis(const double* X, int64_t m, int64_t c, double delta, Buf& core, int* r_out, StageClock& clk,
                             int k, cudaStream_t s, double stop_frac = 0.03) {
  std::vector<SvdPart> parts(1);
  parts[0].X = X;
  parts[0].m = m;
  parts[0].c = c;
  PTTK_TRY(svd_factor(parts, delta, stop_frac, clk, k, s));
  std::vector<int> perm;
  parts[0].r = truncation(parts[0].sigma, delta, perm, parts[0].tail2);
  PTTK_TRY(svd_finish(parts, clk, k, s));
  *r_out = parts[0].r;
  core = std::move(parts[0].core);
  return PTTK_OK;
}

// Packs device cores (core k: ranks[k] x n x ranks[k+1], column-major) into the handle.
static pttk_status pack_cores(pttk_tt* tt, std::vector<Buf>& cores, cudaStream_t s) {
  size_t off = 0;
  for (int k = 0; k < tt->D; ++k) {
    tt->core_off[k] = off;
    off += tt->core_elems(k);
  }
  tt->core_total = off;
  PTTK_CUDA(cudaMalloc(&tt->cores64, sizeof(double) * off));
  PTTK_CUDA(cudaMalloc(&tt->cores32, sizeof(float) * off));
  for (int k = 0; k < tt->D; ++k)
    PTTK_CUDA(cudaMemcpyAsync(tt->cores64 + tt->core_off[k], cores[k].p,
                              sizeof(double) * tt->core_elems(k), cudaMemcpyDeviceToDevice, s));
  cast_f32_kernel<<<grid1d((int64_t)off, 256), 256, 0, s>>>(tt->cores64, (int64_t)off, tt->cores32); pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  PTTK_CUDA(cudaStreamSynchronize(s));
  return PTTK_OK;
}

// squared Frobenius norm of x (n doubles), synchronous
static pttk_status sumsq_host(const double* x, int64_t n, double* out, cudaStream_t s) {
  Buf part, scal;
  const unsigned nb = grid1d(n, 256, 4);
  PTTK_TRY(part.alloc(nb, s));
  PTTK_TRY(scal.alloc(1, s));
  sumsq_kernel<<<nb, 256, 0, s>>>(x, n, part.p); pttk::count_launch();
  sum_kernel<<<1, 256, 0, s>>>(part.p, (int)nb, scal.p); pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  PTTK_CUDA(cudaMemcpyAsync(out, scal.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  PTTK_CUDA(cudaStreamSynchronize(s));
  return PTTK_OK;
}

// ---------------- parity sectors ------------------------------------------------------------------
namespace {

// *bad |= bit s if some nonzero entry of C has indices of different parity in modes s and d + dth + s
__global__ void __launch_bounds__(256) find_sectors_kernel(const double* __restrict__ C, int64_t total, int n, int d, int dth,
                                                           unsigned* __restrict__ bad) {
  unsigned mine = 0;
  const unsigned all = (1u << d) - 1u;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    if (C[e] == 0.0) continue;  // a NaN counts as nonzero
    uint32_t q = (uint32_t)e;   // total <= 4e9 < 2^32
    unsigned px = 0, py = 0;
    for (int j = 0; j < d; ++j, q /= n) px |= ((q % n) & 1u) << j;
    for (int j = 0; j < dth; ++j) q /= n;
    for (int j = 0; j < d; ++j, q /= n) py |= ((q % n) & 1u) << j;
    mine |= px ^ py;
    if (mine == all) break;
  }
  for (int o = 16; o; o >>= 1) mine |= __shfl_xor_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0 && mine) atomicOr(bad, mine);
}

// The columns of one sector of an unfolding: the remaining modes in order, those of y_s (s a symmetric dimension)
// with ceil(n / 2) values h standing for index 2 h + parity, where the parity is the sector's bit, flipped by
// the parity of x_s's index if x_s is among the remaining modes.
struct SectorCols {
  int nd, n;
  int ext[PTTK_MAX_D];
  int xs[PTTK_MAX_D];   // -2: a whole mode; -1: halved; >= 0: halved, with x_s at that position
  int bit[PTTK_MAX_D];  // the sector's bit of a halved mode
};
// Column index in the whole unfolding, or -1 where n is odd and the last half index falls outside.
__device__ __forceinline__ int64_t sector_col(const SectorCols& sc, uint32_t cc) {
  int64_t col = 0, st = 1;
  unsigned odd = 0;  // parity of the index at each position
  bool in = true;
  for (int t = 0; t < sc.nd; ++t) {
    int v = (int)(cc % (uint32_t)sc.ext[t]);
    cc /= (uint32_t)sc.ext[t];
    if (sc.xs[t] > -2) {
      v = 2 * v + (sc.bit[t] ^ (sc.xs[t] >= 0 ? (int)(odd >> sc.xs[t] & 1u) : 0));
      in = in && v < sc.n;
    }
    odd |= (unsigned)(v & 1) << t;
    col += v * st;
    st *= sc.n;
  }
  return in ? col : -1;
}

// XQ (mq x cs) = rows `rows` and the sector's columns of X (m rows); one warp per column
__global__ void __launch_bounds__(256) gather_sector_kernel(const double* __restrict__ X, int64_t m, const int* __restrict__ rows,
                                                            int mq, SectorCols sc, int64_t cs, double* __restrict__ XQ) {
  const int lane = threadIdx.x & 31;
  for (int64_t cc = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; cc < cs; cc += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t col = sector_col(sc, (uint32_t)cc);
    for (int i = lane; i < mq; i += 32) XQ[i + mq * cc] = col < 0 ? 0.0 : X[rows[i] + m * col];
  }
}
// X[ids[l] + r col] = YQ[l + rq cc] (X: r rows)
__global__ void __launch_bounds__(256) scatter_sector_kernel(const double* __restrict__ YQ, int rq, const int* __restrict__ ids,
                                                             int64_t r, SectorCols sc, int64_t cs, double* __restrict__ X) {
  const int lane = threadIdx.x & 31;
  for (int64_t cc = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; cc < cs; cc += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    const int64_t col = sector_col(sc, (uint32_t)cc);
    if (col < 0) continue;
    for (int l = lane; l < rq; l += 32) X[ids[l] + r * col] = YQ[l + rq * cc];
  }
}
// G[rows[i] + m ids[l]] = core[i + mq l]
__global__ void __launch_bounds__(256) scatter_core_kernel(const double* __restrict__ core, const int* __restrict__ rows, int mq,
                                                           const int* __restrict__ ids, int rq, int64_t m, double* __restrict__ G) {
  const int64_t total = (int64_t)mq * rq;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x)
    G[rows[e % mq] + m * ids[e / mq]] = core[e];
}

}  // namespace

pttk_status tt_svd_run(pttk_tt* tt, double* X, double tol, cudaStream_t s) {
  const int D = tt->D, n = tt->n, d = tt->d, dth = tt->dtheta;
  StageClock clk(s);
  int64_t total = 1;
  for (int k = 0; k < D; ++k) total *= n;

  // ||C||_F
  double sumsq = 0.0;
  PTTK_TRY(sumsq_host(X, total, &sumsq, s));
  const double delta = tol / sqrt((double)(D - 1)) * sqrt(sumsq);
  // dimensions whose parities agree in every nonzero entry
  unsigned bad = 0;
  {
    Buf flag;
    PTTK_TRY(flag.alloc(1, s));
    PTTK_CUDA(cudaMemsetAsync(flag.p, 0, sizeof(double), s));
    find_sectors_kernel<<<grid1d(total, 256), 256, 0, s>>>(X, total, n, d, dth, reinterpret_cast<unsigned*>(flag.p)); pttk::count_launch();
    PTTK_CUDA(cudaMemcpyAsync(&bad, flag.p, sizeof bad, cudaMemcpyDeviceToHost, s));
    PTTK_CUDA(cudaStreamSynchronize(s));
  }
  const unsigned sym = ~bad & ((1u << d) - 1u);
  // charge of index v of mode k
  auto charge = [&](int k, int v) -> unsigned {
    const int dim = k < d ? k : k >= d + dth ? k - d - dth : -1;
    return dim >= 0 && (sym >> dim & 1u) ? (unsigned)(v & 1) << dim : 0u;
  };

  std::vector<Buf> cores(D);
  tt->ranks[0] = 1;
  int64_t r_prev = 1;
  std::vector<unsigned> qa(1, 0u);  // charges of the bond's values
  const double* cur = X;
  Buf kept;  // the tensor after the first step, in cur
  int64_t cur_elems = total;
  for (int k = 0; k < D - 1; ++k) {
    const int64_t m = r_prev * n;
    const int64_t c = cur_elems / m;
    // rows by sector
    std::vector<std::vector<int>> rows(8);
    for (int v = 0; v < n; ++v)
      for (int64_t al = 0; al < r_prev; ++al) rows[qa[al] ^ charge(k, v)].push_back((int)(al + r_prev * v));
    std::vector<SvdPart> parts;
    std::vector<unsigned> sector;
    std::vector<SectorCols> cols;
    std::vector<Buf> XQ, drows;
    int64_t cs = 1;
    for (unsigned q = 0; q < 8; ++q) {
      if (rows[q].empty()) continue;
      // a dimension with neither mode left has charge 0 in every column
      bool any = true;
      for (int t = 0; t < d; ++t)
        if ((sym >> t & 1u) && d + dth + t <= k && (q >> t & 1u)) any = false;
      if (!any) continue;
      SectorCols sc{};
      sc.nd = D - 1 - k;
      sc.n = n;
      cs = 1;
      for (int t = 0; t < sc.nd; ++t) {
        const int mode = k + 1 + t, dim = mode - d - dth;
        sc.ext[t] = n;
        sc.xs[t] = -2;
        if (dim >= 0 && (sym >> dim & 1u)) {
          sc.ext[t] = (n + 1) / 2;
          sc.xs[t] = dim > k ? dim - k - 1 : -1;
          sc.bit[t] = (int)(q >> dim & 1u);
        }
        cs *= sc.ext[t];
      }
      parts.emplace_back();
      SvdPart& pt = parts.back();
      pt.m = (int64_t)rows[q].size();
      pt.c = cs;
      sector.push_back(q);
      cols.push_back(sc);
      XQ.emplace_back();
      drows.emplace_back();
      if (sym == 0) {
        pt.X = cur;
        continue;
      }
      PTTK_TRY(drows.back().alloc_ints(pt.m, s));
      PTTK_CUDA(cudaMemcpyAsync(drows.back().ints(), rows[q].data(), sizeof(int) * pt.m, cudaMemcpyHostToDevice, s));
      PTTK_TRY(XQ.back().alloc(pt.m * cs, s));
      gather_sector_kernel<<<grid1d(cs * 32, 256), 256, 0, s>>>(cur, m, drows.back().ints(), (int)pt.m, sc, cs, XQ.back().p); pttk::count_launch();
      pt.X = XQ.back().p;
    }
    PTTK_CUDA(cudaGetLastError());
    PTTK_TRY(svd_factor(parts, delta, 0.03, clk, k, s));
    // the sectors' singular values are those of the unfolding: one truncation
    std::vector<double> sigma;
    std::vector<int> from;
    double tail2 = 0.0;
    for (size_t i = 0; i < parts.size(); ++i) {
      sigma.insert(sigma.end(), parts[i].sigma.begin(), parts[i].sigma.end());
      from.insert(from.end(), parts[i].sigma.size(), (int)i);
      tail2 += parts[i].tail2;
    }
    std::vector<int> order;
    const int r = truncation(sigma, delta, order, tail2);
    if (clk.on) {
      double t = tail2;
      for (int i = (int)sigma.size() - 1; i >= r; --i) t += sigma[order[i]] * sigma[order[i]];
      const double sr = sigma[order[r - 1]];
      fprintf(stderr, "pttk: tt-svd step %d rank %d: tail^2 / delta^2 at r %.6f, at r - 1 %.6f, ||R22||^2 %.6f\n", k + 1, r, t / (delta * delta),
              (t + sr * sr) / (delta * delta), tail2 / (delta * delta));
    }
    std::vector<std::vector<int>> ids(parts.size());
    std::vector<unsigned> qn(r);
    for (int a = 0; a < r; ++a) {
      const int i = from[order[a]];
      ids[i].push_back(a);
      qn[a] = sector[i];
    }
    for (size_t i = 0; i < parts.size(); ++i) parts[i].r = (int)ids[i].size();
    PTTK_TRY(svd_finish(parts, clk, k, s));
    // G_k, and X <- G_k^T X (r x c), allocated only now that the QR inputs are gone: the sectors of an odd n are a little
    // larger than the tensor's nonzero part, and both with the result took more than the two tensors of whole unfoldings
    Buf nxt;
    PTTK_TRY(nxt.alloc((int64_t)r * c, s));
    if (sym == 0) {
      cores[k] = std::move(parts[0].core);
      dgemm(true, false, r, c, m, 1.0, cores[k].p, m, cur, m, 0.0, nxt.p, r, s);
    } else {
      PTTK_TRY(cores[k].alloc(m * r, s));
      PTTK_CUDA(cudaMemsetAsync(cores[k].p, 0, sizeof(double) * m * r, s));
      PTTK_CUDA(cudaMemsetAsync(nxt.p, 0, sizeof(double) * r * c, s));
      for (size_t i = 0; i < parts.size(); ++i) {
        SvdPart& pt = parts[i];
        if (pt.r == 0) continue;
        Buf dids, Y;
        PTTK_TRY(dids.alloc_ints(pt.r, s));
        PTTK_CUDA(cudaMemcpyAsync(dids.ints(), ids[i].data(), sizeof(int) * pt.r, cudaMemcpyHostToDevice, s));
        scatter_core_kernel<<<grid1d(pt.m * pt.r, 256), 256, 0, s>>>(pt.core.p, drows[i].ints(), (int)pt.m, dids.ints(), pt.r, m, cores[k].p); pttk::count_launch();
        PTTK_TRY(Y.alloc(pt.r * pt.c, s));
        dgemm(true, false, pt.r, pt.c, pt.m, 1.0, pt.core.p, pt.m, pt.X, pt.m, 0.0, Y.p, pt.r, s);
        scatter_sector_kernel<<<grid1d(pt.c * 32, 256), 256, 0, s>>>(Y.p, pt.r, dids.ints(), r, cols[i], pt.c, nxt.p); pttk::count_launch();
      }
      PTTK_CUDA(cudaStreamSynchronize(s));  // the host index lists have been read
    }
    PTTK_CUDA(cudaGetLastError());
    clk.mark(k, "project");
    if (clk.on) fprintf(stderr, "pttk: tt-svd step %d rank %d\n", k + 1, r);
    tt->ranks[k + 1] = r;
    kept = std::move(nxt);
    cur = kept.p;
    cur_elems = (int64_t)r * c;
    r_prev = r;
    qa = qn;
  }
  tt->ranks[D] = 1;
  // last core: the remainder (r_{D-1} x n)
  PTTK_TRY(cores[D - 1].alloc(r_prev * n, s));
  PTTK_CUDA(cudaMemcpyAsync(cores[D - 1].p, cur, sizeof(double) * r_prev * n,
                            cudaMemcpyDeviceToDevice, s));
  return pack_cores(tt, cores, s);
}

// TT-Round (Algorithm 1): right-to-left orthogonalisation, then a left-to-right sweep of
// truncated SVDs with delta = tol / sqrt(D-1) ||X||_F. Each factorisation is svd_basis: with
// delta = 0 for the orthogonalisation (an orthonormal basis of the whole range, in place of the
// thin QR; any orthonormal factor serves), with delta for the truncation. Works on device cores
// G[k] (r[k] x nm[k] x r[k+1], column-major) of any mode sizes nm[k]; on return G and r hold the
// rounded TT.
// TT-Round's QR stops at 1e-4 delta (the TT-SVD's at 0.03 delta): its unfoldings are small
// (r_{i-1} n x r_i), so the later stop costs little, and the kept subspaces then agree with
// an exact SVD's to about 1e-4 delta.
constexpr double kRoundStopFrac = 1e-4;

pttk_status tt_round_cores(std::vector<Buf>& G, std::vector<int64_t>& r, const std::vector<int64_t>& nm, double tol,
                           cudaStream_t s) {
  const int D = (int)G.size();
  StageClock clk(s);
  std::vector<Buf> nb(D);
  Buf A, W, T;
  // right to left: (G_i^{1})^T = U W, G_i <- U^T, G_{i-1} <- G_{i-1} x_3 W^T
  for (int i = D - 1; i >= 1; --i) {
    const int64_t m = nm[i] * r[i + 1], c = r[i];
    PTTK_TRY(A.alloc(m * c, s));
    dim3 tg((unsigned)((m + 31) / 32), (unsigned)((c + 31) / 32));
    transpose_kernel<<<tg, dim3(32, 8), 0, s>>>(G[i].p, c, m, nullptr, A.p); pttk::count_launch();
    int k = 0;
    PTTK_TRY(svd_basis(A.p, m, c, 0.0, nb[i], &k, clk, i, s));
    PTTK_TRY(W.alloc((int64_t)k * c, s));
    dgemm(true, false, k, c, m, 1.0, nb[i].p, m, A.p, m, 0.0, W.p, k, s);   // W = U^T A (k x c)
    PTTK_TRY(G[i].alloc((int64_t)k * m, s));
    dim3 tg2((unsigned)((k + 31) / 32), (unsigned)((m + 31) / 32));
    transpose_kernel<<<tg2, dim3(32, 8), 0, s>>>(nb[i].p, m, k, nullptr, G[i].p); pttk::count_launch();
    const int64_t mp = r[i - 1] * nm[i - 1];                               // G_{i-1}^{2}: mp x c
    PTTK_TRY(T.alloc(mp * k, s));
    dgemm(false, true, mp, k, c, 1.0, G[i - 1].p, mp, W.p, k, 0.0, T.p, mp, s);
    std::swap(G[i - 1].p, T.p);
    r[i] = k;
  }
  double sumsq = 0.0;
  PTTK_TRY(sumsq_host(G[0].p, r[0] * nm[0] * r[1], &sumsq, s));
  const double delta = D > 1 ? tol / sqrt((double)(D - 1)) * sqrt(sumsq) : 0.0;
  // left to right: G_i^{2} = U W (truncated), G_i <- U, G_{i+1} <- W x_1 G_{i+1}
  for (int i = 0; i < D - 1; ++i) {
    const int64_t m = r[i] * nm[i], c = r[i + 1];
    int k = 0;
    PTTK_TRY(svd_basis(G[i].p, m, c, delta, nb[i], &k, clk, i, s, kRoundStopFrac));
    PTTK_TRY(W.alloc((int64_t)k * c, s));
    dgemm(true, false, k, c, m, 1.0, nb[i].p, m, G[i].p, m, 0.0, W.p, k, s);
    std::swap(G[i].p, nb[i].p);
    const int64_t cn = nm[i + 1] * r[i + 2];                               // G_{i+1}^{1}: c x cn
    PTTK_TRY(T.alloc((int64_t)k * cn, s));
    dgemm(false, false, k, cn, c, 1.0, W.p, k, G[i + 1].p, c, 0.0, T.p, k, s);
    std::swap(G[i + 1].p, T.p);
    r[i + 1] = k;
  }
  PTTK_CUDA(cudaStreamSynchronize(s));
  return PTTK_OK;
}

pttk_status tt_round_run(const pttk_tt* in, double tol, pttk_tt* out, cudaStream_t s) {
  const int D = in->D;
  std::vector<Buf> G(D);
  std::vector<int64_t> r(D + 1), nm(D, in->n);
  for (int k = 0; k <= D; ++k) r[k] = in->ranks[k];
  for (int k = 0; k < D; ++k) {
    PTTK_TRY(G[k].alloc(in->core_elems(k), s));
    PTTK_CUDA(cudaMemcpyAsync(G[k].p, in->cores64 + in->core_off[k], sizeof(double) * in->core_elems(k),
                              cudaMemcpyDeviceToDevice, s));
  }
  PTTK_TRY(tt_round_cores(G, r, nm, tol, s));
  for (int k = 0; k <= D; ++k) out->ranks[k] = (int)r[k];
  return pack_cores(out, G, s);
}

// Phase 4 of Algorithm 2: TT-Round of [T^(1)(S), G_{d+1}, .., G_{d+d_theta}, T^(3)(T^T)]
// (Eq. twist). Scol: N_s x r_s column-major (the first core 1 x N_s x r_s); theta cores
// ranks[j] x n x ranks[j+1], j < d_theta (ranks[0] = r_s, ranks[d_theta] = r_t); Tt: r_t x N_t
// column-major (the last core r_t x N_t x 1, i.e. T row-major). Inputs are not modified. On
// return out[0] (N_s x r_s' column-major), out[1 .. d_theta] (the rounded theta cores) and
// out[d_theta + 1] (r_t' x N_t column-major) are blocks of the workspace pool that the caller frees with cudaFreeAsync on `s`
// (and copies what it keeps), and new_ranks[0 .. d_theta] their ranks. Synchronises `s`.
pttk_status phase4_round(const double* Scol, int64_t Ns, const double* const* theta_cores, const int* ranks, int n,
                         int dtheta, const double* Tt, int64_t Nt, double tol, double** out, int* new_ranks,
                         cudaStream_t s) {
  const int D = dtheta + 2;
  std::vector<Buf> G(D);
  std::vector<int64_t> r(D + 1), nm(D, n);
  r[0] = 1;
  for (int j = 0; j <= dtheta; ++j) r[j + 1] = ranks[j];
  r[D] = 1;
  nm[0] = Ns;
  nm[D - 1] = Nt;
  for (int k = 0; k < D; ++k) {
    const int64_t e = r[k] * nm[k] * r[k + 1];
    PTTK_TRY(G[k].alloc(e, s));
    const double* src = k == 0 ? Scol : k == D - 1 ? Tt : theta_cores[k - 1];
    PTTK_CUDA(cudaMemcpyAsync(G[k].p, src, sizeof(double) * e, cudaMemcpyDeviceToDevice, s));
  }
  PTTK_TRY(tt_round_cores(G, r, nm, tol, s));
  for (int k = 0; k < D; ++k) {
    out[k] = G[k].p;
    G[k].p = nullptr;
  }
  for (int j = 0; j <= dtheta; ++j) new_ranks[j] = (int)r[j + 1];
  return PTTK_OK;
}

// Orthonormal basis of the range of X (m x c, column-major, not modified): svd_basis with
// delta = 0. *basis is allocated here (cudaMalloc, m x r column-major, r <= min(m, c)); the
// caller frees it with cudaFree. Synchronises `s`.
pttk_status range_basis(const double* X, int64_t m, int64_t c, double** basis, int* r, cudaStream_t s) {
  StageClock clk(s);
  Buf core;
  PTTK_TRY(svd_basis(X, m, c, 0.0, core, r, clk, 0, s));
  // a copy of its own: cudaFree waits for work that still reads it, and does not for scratch of the pool
  PTTK_CUDA(cudaMalloc(basis, sizeof(double) * std::max<int64_t>(m * *r, 1)));
  PTTK_CUDA(cudaMemcpyAsync(*basis, core.p, sizeof(double) * m * *r, cudaMemcpyDeviceToDevice, s));
  return PTTK_OK;
}

// One-sided Jacobi on the columns of A (rows x ncols, column-major), in place: on return the
// columns are orthogonal, A V = U Sigma. Synchronises `s`.
pttk_status jacobi_columns(double* A, int64_t rows, int ncols, cudaStream_t s) {
  return jacobi_batch({Jac{A, rows, ncols}}, s);
}

// FP32 tensor -> FP64 work buffer
pttk_status widen_to_f64(const float* in, int64_t n, double* out, cudaStream_t s) {
  widen_f32_kernel<<<grid1d(n, 256), 256, 0, s>>>(in, n, out); pttk::count_launch();
  PTTK_CUDA(cudaGetLastError());
  return PTTK_OK;
}

}  // namespace pttk
