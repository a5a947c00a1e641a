// Small dense linear algebra of the bond update, FP64 unless noted.
//
//   k_env_factor   pivoted Cholesky square root L of a message M (L^T L = M):
//                  the environment square root of Sec. 2.5 step 1 (Fig. 1
//                  "pseudo_sqrt"); any factor with L^T L = M gives the same cv
//                  Gram, so no eigensolver is needed.
//   k_branch       Eq. 10 branch rule: Cholesky-QR when n > n_thr and
//                  m / n > ratio_thr, the other branch otherwise (Sec. 4.2).
//   k_hh_level     FP64 storage: Householder QR (TSQR tree, R only) of cv
//                  (Sec. 4.2 Householder-QR); each tree block factored in panels
//                  (compact WY).  FP32 storage forms the exact Gram of cv instead
//                  (k_gram_exact) and factors that.
//   k_form         fold the gate's operator-Schmidt factors into the
//                  R-factor: X = (F_kappa (x) 1) cv, G = X^T X or B = R-side of X.
//   k_factor       rank-revealing factor T of X: pivoted Cholesky of G (from a
//                  Gram) or column-pivoted Householder of B (from an R-factor).
//   k_core         per bond: R1 R2^T, one-sided Jacobi SVD, truncation
//                  (Eq. 11), lambda (Eq. 12), reconstruct matrices W1, W2
//                  (Sec. 2.5 steps 5-8 in Q-less form), messages diag(lambda).
//   k_env_eig      eigenbasis and square roots of a message (BP rotations).
//   k_rotate_back  a Gram of the rotated tensor back into the bond's basis.
#include <algorithm>
#include <cstddef>
#include <type_traits>

#include "kernels.h"
#include "linalg.h"

namespace pepo {

// ------------------------------------------------------------ block helpers
__device__ inline double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// An FP64 operation of a warp holds its quarter of the SM's FP64 units for 64
// clocks, whatever the number of useful lanes: scalars that the whole block needs (a root, a quotient, the sum
// of the warps' partials) are formed by one warp and read from shared memory, and
// magnitudes are compared as integers.

// x 2^(1023 - e), e >= x's biased exponent, cut to 24 bits; (double)x of a normal
// number or zero: by integer operations
__device__ __forceinline__ float top_float(double x, int e) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int ex = (hi >> 20) & 0x7ff, f = ex - e + 127;
  const int bits = (hi & 0x80000000) | (f << 23) | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29);
  return ex == 0 || f <= 0 ? 0.f : __int_as_float(bits);
}
__device__ __forceinline__ double wide(float x) {
  const int b = __float_as_int(x);
  return (b & 0x7fffffff) == 0 ? 0.0
                               : __hiloint2double((b & 0x80000000) | (((b & 0x7fffffff) >> 3) + (896 << 20)), b << 29);
}

// Block-wide sum; `red` must hold 32 doubles.  All threads return it.
__device__ inline double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = lane < nw ? red[lane] : 0.0;
    t = warp_sum(t);
    __syncwarp();
    if (lane == 0) red[0] = t;
  }
  __syncthreads();
  return red[0];
}

// Order of a magnitude (>= 0) as an integer; NaN and negative values below every number.
__device__ __forceinline__ long long mag_key(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0 && b <= 0x7ff0000000000000ll ? b : (b == (long long)0x8000000000000000ull ? 0ll : -1ll);
}

// Block-wide argmax over values[i] for i in [lo, hi) (hi > lo); returns the
// index (smallest index among ties), always inside [lo, hi): lo when no value
// is a number >= 0, where the callers' pivot test then stops.  `rk` needs 32
// long longs, `ri` 32 ints.
__device__ inline int block_argmax(const double* values, int lo, int hi, long long* rk, int* ri) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  long long best = -1;
  int bi = hi;
  for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) {
    const long long x = mag_key(values[i]);
    if (x > best) { best = x; bi = i; }
  }
  auto fold = [&]() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
  };
  fold();
  if (lane == 0) { rk[w] = best; ri[w] = bi; }
  __syncthreads();
  if (w == 0) {
    best = lane < nw ? rk[lane] : -1;
    bi = lane < nw ? ri[lane] : hi;
    fold();
    __syncwarp();
    if (lane == 0) ri[0] = bi;
  }
  __syncthreads();
  const int idx = ri[0];
  __syncthreads();
  return idx < hi ? idx : lo;
}

// =============================================================== env factor
// Pivoted (outer-product) Cholesky of the symmetrised message in shared memory.
__global__ void __launch_bounds__(256)
k_env_factor(const EnvFactorItem* __restrict__ items, int* ival) {
  const EnvFactorItem it = items[blockIdx.x];
  const double rel = it.rel;
  const int n = ival[it.chi_idx];
  extern __shared__ __align__(16) double sm[];
  double* A = sm;                 // n x n
  double* dg = A + n * n;         // n
  int* perm = reinterpret_cast<int*>(dg + n);
  __shared__ long long rv[32];
  __shared__ int ri[32];
  __shared__ double sh_r[2];
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    int i = e / n, j = e - i * n;
    A[e] = 0.5 * (it.M[i * it.ld + j] + it.M[j * it.ld + i]);
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) perm[i] = i;
  __syncthreads();
  double d0 = 0.0;
  int rank = n;
  for (int j = 0; j < n; ++j) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dg[i] = (i >= j) ? A[i * n + i] : -1.0;
    __syncthreads();
    int p = block_argmax(dg, j, n, rv, ri);
    double dp = dg[p];
    if (j == 0) d0 = dp;
    if (!(dp > rel * d0) || !(dp > 0.0)) { rank = j; break; }
    if (p != j) {  // symmetric swap of rows/cols j and p
      for (int k = threadIdx.x; k < n; k += blockDim.x) {
        double t = A[j * n + k]; A[j * n + k] = A[p * n + k]; A[p * n + k] = t;
      }
      __syncthreads();
      for (int k = threadIdx.x; k < n; k += blockDim.x) {
        double t = A[k * n + j]; A[k * n + j] = A[k * n + p]; A[k * n + p] = t;
      }
      if (threadIdx.x == 0) { int t = perm[j]; perm[j] = perm[p]; perm[p] = t; }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      sh_r[0] = sqrt(A[j * n + j]);
      sh_r[1] = 1.0 / sh_r[0];
    }
    __syncthreads();
    const double inv = sh_r[1];
    for (int k = j + 1 + threadIdx.x; k < n; k += blockDim.x) A[j * n + k] *= inv;
    if (threadIdx.x == 0) A[j * n + j] = sh_r[0];
    __syncthreads();
    for (int a = j + 1 + (int)(threadIdx.x >> 5); a < n; a += (int)(blockDim.x >> 5)) {
      const double x = A[j * n + a];
      for (int b = j + 1 + (int)(threadIdx.x & 31); b < n; b += 32) A[a * n + b] -= x * A[j * n + b];
    }
    __syncthreads();
  }
  // L[a][perm[q]] = R[a][q] (upper part), rows a < rank
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    int a = e / n, q = e - a * n;
    double v = (a < rank && q >= a) ? A[a * n + q] : 0.0;
    it.L[a * it.ld + perm[q]] = v;
  }
  if (threadIdx.x == 0) ival[it.rank_idx] = rank;
}

cudaError_t launch_env_factor(const EnvFactorItem* items, int n_items, int chimax, int* ival,
                              cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  size_t smem = sizeof(double) * ((size_t)chimax * chimax + chimax) + sizeof(int) * chimax;
  cudaError_t e = cudaFuncSetAttribute(k_env_factor, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  k_env_factor<<<n_items, 256, smem, s>>>(items, ival);
  return cudaGetLastError();
}

// =================================================================== branch
__device__ inline void cv_shape(const TView& v, const int* ival, long long& m, int& n) {
  m = 1;
  for (int k = 0; k + 1 < v.nlegs; ++k) m *= ival[v.dim[k]];
  n = 4 * (v.nlegs > 0 ? ival[v.dim[v.nlegs - 1]] : 1);
}

__global__ void k_branch(const SiteFacItem* __restrict__ items, int n_items, int* ival) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_items) return;
  const SiteFacItem it = items[i];
  long long m;
  int n;
  cv_shape(it.cv, ival, m, n);
  ival[it.branch_idx] = (n > it.n_thr && (double)m / (double)n > it.ratio_thr) ? 1 : 0;
}

cudaError_t launch_branch(const SiteFacItem* items, int n_items, int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  k_branch<<<ceil_div(n_items, 128), 128, 0, s>>>(items, n_items, ival);
  return cudaGetLastError();
}

// ========================================================== Householder TSQR
// FP64 storage (FP32 storage factors the exact Gram of its data, k_gram_exact).
// Leaf rows L = max(4n, 128).  Level 0 factors each leaf in place; level l >= 1
// gathers the R-blocks of four level-(l-1) blocks into the first one and
// factors the stack.  R replaces the top rows of the block; entries below the
// diagonal are zeroed (Q is never needed: the update is Q-less).
__host__ __device__ inline long long hh_leaf_rows(int n) { return n * 4 > kHhLeafRows ? (long long)n * 4 : kHhLeafRows; }
constexpr int kHhThreads = 512;   // threads of a TSQR block

// Panel width of the blocked QR: the panel (L x NB) lives in shared memory.
constexpr int kHhPanel = 8;

// Shared-memory plan of one TSQR block (leaf rows L): panel V (column-major,
// leading dimension L + 1 so that consecutive rows of a column and the rows
// of consecutive columns fall in different banks), per-warp partial products
// of the trailing update, W = V^T A and W2 = T^T W, V^T V, and per reflection
// tau and the scale of its vector.
struct HhSmem {
  size_t p, red, wd, w2, vtv, tau, inv, total;
  int lp;
};
__host__ __device__ inline HhSmem hh_smem(long long L) {
  constexpr int NB = kHhPanel;
  HhSmem m;
  m.lp = (int)L + 1;
  size_t o = 0;
  m.p = o;    o += sizeof(double) * (size_t)NB * m.lp;
  o = (o + 15) & ~(size_t)15;
  m.red = o;  o += sizeof(double) * (size_t)(kHhThreads / 32) * NB * 32;
  m.wd = o;   o += sizeof(double) * (size_t)NB * 32;
  m.w2 = o;   o += sizeof(double) * (size_t)NB * 32;
  m.vtv = o;  o += sizeof(double) * (size_t)NB * NB;
  m.tau = o;  o += sizeof(double) * (size_t)NB;
  m.inv = o;  o += sizeof(double) * (size_t)NB;
  m.total = o;
  return m;
}

__device__ inline void ld4(const double* p, double (&x)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
}
__device__ inline void st4(double* p, const double (&x)[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(x[0], x[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(x[2], x[3]);
}

// The reflection that takes a column with diagonal alpha and squared norm s (diagonal
// included) to beta e_1: v = (1, inv x), H = 1 - tau v v^T.  1 / sqrt(s) and the
// reciprocal come from FP32 seeds by one cubic step each (a library root and two
// quotients take ~25 FP64 operations, this takes 11); tau = 1 - alpha / beta needs
// no quotient.
__device__ inline void reflector(double alpha, double s, double& beta, double& tau, double& inv) {
  beta = alpha;
  tau = 0.0;
  inv = 1.0;
  if (!(s > 0.0)) return;
  const int es = (__double2hiint(s) >> 20) & 0x7ff;
  if (es < 2 || es >= 0x7ff) {                              // subnormal, infinite or NaN
    const double norm = sqrt(s);
    beta = alpha >= 0.0 ? -norm : norm;
    inv = 1.0 / (alpha - beta);
    tau = (beta - alpha) / beta;
    return;
  }
  const int k = (es - 1023) >> 1;                           // s = m 4^k, m in [1, 4)
  const double m = __hiloint2double(__double2hiint(s) - k * (1 << 21), __double2loint(s));
  const double y0 = wide(rsqrtf(top_float(m, 1024) * 2.f));
  const double e = fma(-m * y0, y0, 1.0);
  const double y = fma(y0 * e, fma(0.375, e, 0.5), y0);     // 1 / sqrt(m)
  const double nm = m * y;
  const double norm = __hiloint2double(__double2hiint(nm) + k * (1 << 20), __double2loint(nm));
  const double a = fabs(alpha);
  tau = fma(__hiloint2double(__double2hiint(y) - k * (1 << 20), __double2loint(y)), a, 1.0);
  beta = alpha >= 0.0 ? -norm : norm;
  const double d = a + norm;                                // |alpha - beta| in [norm, 2 norm]
  const int ed = (__double2hiint(d) >> 20) & 0x7ff;
  double z = wide(__frcp_rn(top_float(d, ed)));             // 2^(ed - 1023) / d
  z = __hiloint2double(__double2hiint(z) - (ed - 1023) * (1 << 20), __double2loint(z));
  const double r = fma(-d, z, 1.0);
  z = fma(fma(r, r, r), z, z);
  inv = alpha >= 0.0 ? z : -z;
}

// Halving exchange: sums the 2 H values of v over the lanes that differ in bit `bit`;
// the lane with the bit clear keeps the first H sums, the other the last H (H
// additions; summing every value on every lane takes 2 H).
template <int H, int N>
__device__ __forceinline__ void halve(double (&v)[N], int bit) {
  const bool up = (threadIdx.x & bit) != 0;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const double send = up ? v[i] : v[i + H], keep = up ? v[i + H] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
  }
}

// One pass of the trailing update over columns cb .. cb + 4 NQ - 1 (those below c0
// stay): A <- A - V W2, W2 = T^T (V^T A).  Lanes: NQ column quads x 32 / NQ row groups.
template <int NQ>
__device__ __forceinline__ void hh_trailing(double* A, int n, int j0, int pr, int nb, int cb, int c0, const double* P,
                                            int lp, double* red, double* Wd, double* W2, const double* VtV,
                                            const double* tau) {
  constexpr int NB = kHhPanel;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = kHhThreads / 32;
  const int kq = tid % NQ, rgi = tid / NQ;
  constexpr int nrg = kHhThreads / NQ;
  const int cq = cb + 4 * kq;
  const bool colok = cq < n;
  double v[NB * 4];
#pragma unroll
  for (int q = 0; q < NB * 4; ++q) v[q] = 0.0;
  if (colok) {
    for (int i = rgi; i < pr; i += nrg) {
      double a[4];
      ld4(A + (long long)(j0 + i) * n + cq, a);
#pragma unroll
      for (int l = 0; l < NB; ++l) {
        const double x = P[l * lp + i];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[l * 4 + q] = fma(x, a[q], v[l * 4 + q]);
      }
    }
  }
  // rows of a warp: each lane ends up with the sums of its share of the 32 values
  halve<16>(v, 16);
  int first = lane & 16 ? 16 : 0;
  halve<8>(v, 8);
  first += lane & 8 ? 8 : 0;
  constexpr int KEEP = NQ;                                  // 32 / (32 / NQ)
  if constexpr (NQ <= 4) { halve<4>(v, 4); first += lane & 4 ? 4 : 0; }
  if constexpr (NQ <= 2) { halve<2>(v, 2); first += lane & 2 ? 2 : 0; }
#pragma unroll
  for (int i = 0; i < KEEP; ++i) {
    const int l = (first + i) >> 2, q = (first + i) & 3;
    red[(warp * NB + l) * 32 + 4 * kq + q] = v[i];
  }
  __syncthreads();
  for (int e = tid; e < NB * 4 * NQ; e += kHhThreads) {
    const int l = e / (4 * NQ), k = e % (4 * NQ);
    double z = 0.0;
#pragma unroll
    for (int w = 0; w < NW; ++w) z += red[(w * NB + l) * 32 + k];
    Wd[l * 32 + k] = z;
  }
  __syncthreads();
  // T^T W by forward substitution: T^-T is V^T V's lower triangle with 1 / tau on the
  // diagonal
  if (tid < 4 * NQ) {
    double w[NB];
#pragma unroll
    for (int l = 0; l < NB; ++l) {
      double z = Wd[l * 32 + tid];
#pragma unroll
      for (int mm = 0; mm < l; ++mm) z = fma(-VtV[mm * NB + l], w[mm], z);
      w[l] = l < nb ? z * tau[l] : 0.0;
      W2[l * 32 + tid] = cb + tid < c0 ? 0.0 : w[l];
    }
  }
  __syncthreads();
  if (colok) {
    double w2[NB][4];
#pragma unroll
    for (int l = 0; l < NB; ++l)
#pragma unroll
      for (int q = 0; q < 4; ++q) w2[l][q] = W2[l * 32 + 4 * kq + q];
    for (int i = rgi; i < pr; i += nrg) {
      double* pa = A + (long long)(j0 + i) * n + cq;
      double a[4];
      ld4(pa, a);
#pragma unroll
      for (int l = 0; l < NB; ++l) {
        const double x = P[l * lp + i];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = fma(-x, w2[l][q], a[q]);
      }
      if (cq < c0) {
        // quad straddling the panel: keep the panel's columns untouched
        double o[4];
        ld4(pa, o);
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (cq + q < c0) a[q] = o[q];
      }
      st4(pa, a);
    }
  }
  __syncthreads();
}

// Householder QR of one TSQR block A (rows x n, row-major, n % 4 == 0, base
// 16-byte aligned) in place: R in the top rows, zeros below (Q is not kept).
// Blocked by panels of NB columns in the compact WY form H_1 ... H_nb =
// I - V T V^T: the panel is factored in shared memory, then the trailing
// columns take all nb reflections in one pass, A <- A - V (T^T (V^T A)),
// instead of one pass per reflection.  512 threads.
//
// Bound: the FP64 units, a quarter of the SM each, one warp operation per 64
// clocks: what counts is the operations of the busiest quarter.  So the warp of
// a panel's next column reflects it, sums its squares and forms its reflection
// in one go, alone on its quarter, while the other columns' warps share the rest
// (one barrier a column); trailing sums are exchanged by halves; the last
// columns take as many lanes as they fill.  Class: 4x4 chi = 12 layer 5.5 -> 3.4 ms, 3x3 chi = 8 evolution
// 5.5 -> 3.4.
__device__ void hh_block_qr(double* A, long long rows, int n, unsigned char* smem, const HhSmem& S) {
  constexpr int NB = kHhPanel;
  double* P = reinterpret_cast<double*>(smem + S.p);
  double* red = reinterpret_cast<double*>(smem + S.red);
  double* Wd = reinterpret_cast<double*>(smem + S.wd);
  double* W2 = reinterpret_cast<double*>(smem + S.w2);
  double* VtV = reinterpret_cast<double*>(smem + S.vtv);
  double* tau = reinterpret_cast<double*>(smem + S.tau);
  double* inv = reinterpret_cast<double*>(smem + S.inv);
  const int lp = S.lp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = kHhThreads / 32;
  const int kmax = (int)(rows < n ? rows : n);
  // column jj of the panel: its reflection from its rows jj .. pr - 1, by a warp
  auto reflect = [&](int jj, int pr) {
    double* col = P + jj * lp;
    double s = 0.0;
    for (int i = jj + lane; i < pr; i += 32) s = fma(col[i], col[i], s);
    s = warp_sum(s);
    double beta, t, z;
    reflector(col[jj], s, beta, t, z);
    __syncwarp();
    if (lane == 0) {
      col[jj] = beta;
      tau[jj] = t;
      inv[jj] = z;
    }
  };
  for (int j0 = 0; j0 < kmax; j0 += NB) {
    const int nb = kmax - j0 < NB ? kmax - j0 : NB;
    const int pr = (int)(rows - j0);
    // ---- panel rows j0.., columns j0..j0+nb-1 (zero columns beyond nb)
    for (int e = tid; e < pr * NB; e += kHhThreads) {
      const int i = e / NB, l = e - i * NB;
      P[l * lp + i] = (l < nb) ? A[(long long)(j0 + i) * n + j0 + l] : 0.0;
    }
    __syncthreads();
    if (warp == 0) reflect(0, pr);
    __syncthreads();
    // ---- unblocked Householder on the panel, its vectors unscaled: x = v / inv
    // below the diagonal.  Column jj + 1 belongs to warp 0, the others to the
    // warps of the other quarters.
    for (int jj = 0; jj + 1 < nb; ++jj) {
      const int c = warp == 0 ? jj + 1 : (warp & 3) == 0 ? nb : jj + 1 + warp - (warp >> 2);
      if (c < nb) {
        const double* col = P + jj * lp;
        double* pc = P + c * lp;
        const double t = tau[jj], z = inv[jj];
        if (t != 0.0) {
          double acc = 0.0;
          for (int i = jj + 1 + lane; i < pr; i += 32) acc = fma(col[i], pc[i], acc);
          acc = warp_sum(acc);
          const double w = t * fma(z, acc, pc[jj]), wz = w * z;
          __syncwarp();
          if (lane == 0) pc[jj] -= w;
          for (int i = jj + 1 + lane; i < pr; i += 32) pc[i] = fma(-wz, col[i], pc[i]);
          __syncwarp();
        }
        if (c == jj + 1) reflect(c, pr);
      }
      __syncthreads();
    }
    // ---- R of the panel and zeros below it back to A; V explicit in P (scaled,
    // unit diagonal, zeros above) for the WY products
    for (int e = tid; e < pr * NB; e += kHhThreads) {
      const int i = e / NB, l = e - i * NB;
      if (l < nb) {
        const double x = P[l * lp + i];
        A[(long long)(j0 + i) * n + j0 + l] = (i <= l) ? x : 0.0;
        P[l * lp + i] = i < l ? 0.0 : i == l ? 1.0 : x * inv[l];
      }
    }
    __syncthreads();
    const int c0 = j0 + nb;
    if (c0 >= n) continue;
    // ---- V^T V above the diagonal
    for (int q = warp; q < NB * NB; q += NW) {
      const int l = q / NB, j = q - l * NB;
      if (l >= j || j >= nb) continue;
      const double* vl = P + l * lp;
      const double* vj = P + j * lp;
      double acc = 0.0;
      for (int i = j + lane; i < pr; i += 32) acc = fma(vl[i], vj[i], acc);
      acc = warp_sum(acc);
      if (lane == 0) VtV[l * NB + j] = acc;
    }
    if (tid < NB * NB && (tid % NB >= nb || tid / NB >= tid % NB)) VtV[tid] = 0.0;
    __syncthreads();
    for (int cb = c0 & ~3; cb < n; cb += 32) {
      if (n - cb > 16) hh_trailing<8>(A, n, j0, pr, nb, cb, c0, P, lp, red, Wd, W2, VtV, tau);
      else if (n - cb > 8) hh_trailing<4>(A, n, j0, pr, nb, cb, c0, P, lp, red, Wd, W2, VtV, tau);
      else hh_trailing<2>(A, n, j0, pr, nb, cb, c0, P, lp, red, Wd, W2, VtV, tau);
    }
  }
}

__global__ void __launch_bounds__(kHhThreads)
k_hh_level(const SiteFacItem* __restrict__ items, int level, void* const* ptrs, const int* ival, int pass) {
  const SiteFacItem it = items[blockIdx.y];
  if (ival[it.branch_idx] != pass) return;
  long long m;
  int n;
  cv_shape(it.cv, ival, m, n);
  const long long L = hh_leaf_rows(n);
  long long nb0 = (m + L - 1) / L;
  // block size in rows at this level, and number of blocks
  long long span = L, nblk = nb0;
  for (int l = 0; l < level; ++l) {
    if (nblk == 1) return;        // already reduced at an earlier level
    span *= 4;
    nblk = (nblk + 3) / 4;
  }
  const long long g = blockIdx.x;
  if (g >= nblk) return;
  double* A = static_cast<double*>(ptrs[it.cv.ref]);
  extern __shared__ __align__(16) unsigned char hh_sh[];
  const HhSmem S = hh_smem(L);            // within the launch's plan for nmax >= n
  double* base = A + g * span * n;
  long long rows;
  if (level == 0) {
    long long r0 = g * span;
    rows = (m - r0) < span ? (m - r0) : span;
  } else {
    // gather the R rows of the four children into the first child's area
    const long long cspan = span / 4;
    rows = 0;
    for (int c = 0; c < 4; ++c) {
      const long long cr0 = g * span + c * cspan;
      if (cr0 >= m) break;
      long long crows_full = (m - cr0) < cspan ? (m - cr0) : cspan;
      // rows of the child's R: min(rows of the child's own stack, n); the stack
      // of a child has at most min(crows_full, ...) rows, and its R at most n
      long long rr = crows_full < n ? crows_full : n;
      if (c > 0) {
        const double* src = A + cr0 * n;                    // the stack (4 n rows) ends before it
        for (long long e = threadIdx.x; e < rr * n; e += blockDim.x) base[rows * n + e] = src[e];
      }
      rows += rr;
    }
    __syncthreads();
  }
  hh_block_qr(base, rows, n, hh_sh, S);
}

cudaError_t launch_hh_level(const SiteFacItem* items, int n_items, int level, int grid_x, int nmax,
                            void* const* ptrs, const int* ival, cudaStream_t s, int pass) {
  if (n_items == 0) return cudaSuccess;
  const size_t smem = hh_smem(hh_leaf_rows(nmax)).total;
  cudaError_t e = cudaFuncSetAttribute(k_hh_level, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  k_hh_level<<<dim3(grid_x, n_items), kHhThreads, smem, s>>>(items, level, ptrs, ival, pass);
  return cudaGetLastError();
}

// R (top min(m, n) rows of cv after the tree) -> FP64 C buffer, rows -> kfac
// acct (2 doubles, may be null): algorithmic FLOPs and bytes of the QR of
// each factored m x n matrix (2 m n^2 - 2 n^3 / 3 for m >= n, else
// 2 m^2 n - 2 m^3 / 3; one read of the matrix), accumulated on the device
// because only the device knows which sites took this branch.
__global__ void k_hh_extract(const SiteFacItem* __restrict__ items, void* const* ptrs, int* ival, int pass,
                             double* acct) {
  const SiteFacItem it = items[blockIdx.x];
  if (ival[it.branch_idx] != pass) return;
  long long m;
  int n;
  cv_shape(it.cv, ival, m, n);
  const int k = (int)(m < n ? m : n);
  if (acct && threadIdx.x == 0) {
    const double dm = (double)m, dn = (double)n;
    const double f = m >= n ? 2.0 * dm * dn * dn - 2.0 * dn * dn * dn / 3.0
                            : 2.0 * dm * dm * dn - 2.0 * dm * dm * dm / 3.0;
    atomicAdd(&acct[0], f);
    atomicAdd(&acct[1], dm * dn * sizeof(double));
  }
  const double* A = static_cast<const double*>(ptrs[it.cv.ref]);
  for (int e = threadIdx.x; e < k * n; e += blockDim.x) {
    int a = e / n, q = e - a * n;
    it.C[(long long)a * it.ldc + q] = (q >= a) ? A[(long long)a * n + q] : 0.0;
  }
  if (threadIdx.x == 0) ival[it.kfac_idx] = k;
}

cudaError_t launch_hh_extract(const SiteFacItem* items, int n_items, void* const* ptrs, int* ival,
                              cudaStream_t s, int pass, double* acct) {
  if (n_items == 0) return cudaSuccess;
  k_hh_extract<<<n_items, 256, 0, s>>>(items, ptrs, ival, pass, acct);
  return cudaGetLastError();
}

// ============================================================ formG / formB
// From a Gram: G[(c,k),(c',k')] = sum_{p,q} (F_k^T F_k')[p,q] C[(c,p),(c',q)].
// From a Householder R: B[(a,p'),(c,k)] = sum_p F_k[p',p] R[a,(c,p)].
__global__ void k_form(const SiteFacItem* __restrict__ items, const int* ival, int only, int householder) {
  const SiteFacItem it = items[blockIdx.y];
  if (only >= 0 && ival[it.branch_idx] != only) return;
  long long m;
  int n;
  cv_shape(it.cv, ival, m, n);
  const int chic = n / 4;
  const int rg = ival[it.rg_idx];
  const int r = rg * chic;
  __shared__ double F[PEPO_RG * 16];
  __shared__ double H[PEPO_RG * PEPO_RG * 16];
  for (int e = threadIdx.x; e < rg * 16; e += blockDim.x) F[e] = it.F[e];
  __syncthreads();
  if (ival[it.branch_idx] == 1 || !householder) {
    for (int e = threadIdx.x; e < rg * rg * 16; e += blockDim.x) {
      int k = e / (rg * 16), rest = e % (rg * 16);
      int k2 = rest / 16, pq = rest % 16, p = pq / 4, q = pq % 4;
      double h = 0.0;
      for (int pp = 0; pp < 4; ++pp) h += F[k * 16 + pp * 4 + p] * F[k2 * 16 + pp * 4 + q];
      H[e] = h;
    }
    __syncthreads();
    double* Gp = it.T + (long long)it.ldt * it.ldt;   // G lies behind T (k_factor writes T from it)
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)chic * chic;
         e += (long long)gridDim.x * blockDim.x) {
      int c = (int)(e / chic), c2 = (int)(e % chic);
      double Cb[16];
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) Cb[p * 4 + q] = it.C[(long long)(c * 4 + p) * it.ldc + c2 * 4 + q];
      for (int k = 0; k < rg; ++k)
        for (int k2 = 0; k2 < rg; ++k2) {
          const double* h = H + (k * rg + k2) * 16;
          double g = 0.0;
#pragma unroll
          for (int pq = 0; pq < 16; ++pq) g += h[pq] * Cb[pq];
          Gp[(long long)(c * rg + k) * it.ldt + c2 * rg + k2] = g;
        }
    }
  } else {
    const int k = ival[it.kfac_idx];
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)k * 4 * r;
         e += (long long)gridDim.x * blockDim.x) {
      int row = (int)(e / r), col = (int)(e % r);
      int a = row / 4, pp = row % 4, c = col / rg, kk = col % rg;
      double b = 0.0;
#pragma unroll
      for (int p = 0; p < 4; ++p) b += F[kk * 16 + pp * 4 + p] * it.C[(long long)a * it.ldc + c * 4 + p];
      it.T[(long long)row * it.ldt + col] = b;
    }
  }
}

cudaError_t launch_form(const SiteFacItem* items, int n_items, int grid_x, const int* ival,
                        cudaStream_t s, int only, int householder) {
  if (n_items == 0) return cudaSuccess;
  k_form<<<dim3(grid_x, n_items), 256, 0, s>>>(items, ival, only, householder);
  return cudaGetLastError();
}

// ------------------------------------------------------------ clusters
// The CTAs that share a site's factor or a bond core meet at the hardware cluster barrier (its
// arrive / wait pair orders their global-memory accesses); a cluster of one
// meets at the block barrier.
struct Cta {
  int rank, size;        // this CTA in its cluster, CTAs in it
  long long tid, nthr;   // this thread among the cluster's threads
};
__device__ __forceinline__ void cta_sync(const Cta& c) {
  if (c.size > 1) {
    asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}

// =================================================================== factor
constexpr int kFacThreads = 512;
constexpr int kFacSlices = 4;

// Shared memory of k_factor: the vectors of the cluster Cholesky (or of the
// Householder QR, FP64 storage), then what is left for the factor itself (a
// CTA's columns of U, or the Householder branch's matrix) when it fits.
struct FacSmem {
  size_t cand, uc, part, dq, oq, pos, perm, v, mat, total;
};
__host__ __device__ inline FacSmem fac_smem(int rmax, int nmax, int householder, int csize) {
  FacSmem m;
  const int w = rmax > nmax ? rmax : nmax;
  size_t o = 0;
  m.cand = o; o += 2 * sizeof(double) * w;
  m.uc = o;   o += sizeof(double) * w;
  m.part = o; o += sizeof(double) * kFacSlices * (size_t)((w + csize - 1) / csize);
  m.dq = o;   o += sizeof(double) * w;
  m.oq = o;   o += sizeof(double) * w;
  m.pos = o;  o += sizeof(int) * (size_t)w;
  m.perm = o; o += sizeof(int) * (size_t)w;
  m.v = o;
  if (householder) o += sizeof(double) * ((size_t)4 * nmax + (size_t)4 * rmax);
  o = (o + 15) & ~(size_t)15;
  m.mat = o;
  const size_t cap = (size_t)216 * 1024;
  const size_t want = householder ? sizeof(double) * (size_t)4 * nmax * rmax
                                  : sizeof(double) * (size_t)w * ((w + csize - 1) / csize);
  o += want < cap - o ? want : cap - o;
  m.total = o;
  return m;
}

// a CTA's candidate for the next pivot
struct Pivot {
  double value, own;     // remaining and original diagonal
  int col;
};

__device__ __forceinline__ unsigned cluster_addr(const void* p, int rank) {   // p's address in CTA `rank`
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
template <typename R> __device__ __forceinline__ R cluster_ld(unsigned a);
template <> __device__ __forceinline__ double cluster_ld<double>(unsigned a) {
  double x;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(a) : "memory");
  return x;
}
template <> __device__ __forceinline__ float cluster_ld<float>(unsigned a) {
  float x;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(a) : "memory");
  return x;
}
template <> __device__ __forceinline__ int cluster_ld<int>(unsigned a) {
  int x;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(x) : "r"(a) : "memory");
  return x;
}

// Pivoted Cholesky of a symmetric n x n matrix A (leading dimension lda, read
// only) in precision R by the CTAs of a cluster; returns the rank (pivots <= rel
// times the first end it), or -1 when an accepted pivot keeps less than `safe`
// of its own column's diagonal (safe < 0: not tested).  CTA k owns the w columns
// from k w on: U[j][c] (j steps, c its column, in shared memory where w n values
// fit) is its part of the upper factor, pos[c] the step at which the column
// became a pivot (-1: never), perm[j] the pivot column of step j.
//
// Left-looking: step j forms only row j, U[j, q] = (A[p_j, q] - sum_l<j U[l, p_j]
// U[l, q]) / U[j, p_j], the sum in four interleaved parts (the same bits for every
// cluster size), and nothing is rewritten (the right-looking form updates the trailing square through L2
// at every step).  Columns stay where they are, so a step moves only the
// candidates: every CTA offers its largest remaining diagonal with that column
// of U, the cluster meets once, and all read the winner's column from its
// shared memory (offers alternate between two buffers, so one meeting per
// step is enough).  Bound: the FP64 pipe, r^3 / 6 multiply-adds at 2 per clock
// and SM, plus ~2 us of meeting and latency per step.
template <typename R>
__device__ int chol_cluster(const double* __restrict__ A, int lda, int n, int w, R* U, const Cta& ct, Pivot* offer,
                            R* offer_u, int ldo, R* uc, R* part, R* dq, R* oq, int* pos, int* perm, double rel,
                            double safe) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int c0 = ct.rank * w;
  const int nl = min(w, n - c0) > 0 ? min(w, n - c0) : 0;
  __shared__ int sh_best;
  __shared__ Pivot sh_win;
  __shared__ int sh_from;
  __shared__ R sh_rs;
  for (int i = tid; i < nl; i += kFacThreads) {
    dq[i] = oq[i] = (R)A[(long long)(c0 + i) * lda + c0 + i];
    pos[i] = -1;
  }
  __syncthreads();
  double d0 = 0.0;
  for (int j = 0; j < n; ++j) {
    Pivot* of = offer + (j & 1);
    R* ofu = offer_u + (j & 1) * ldo;
    if (tid < 32) {
      // this CTA's largest remaining diagonal (smallest column among ties; none
      // when every candidate is NaN)
      long long best = -1;
      int bi = n;
      for (int i = lane; i < nl; i += 32)
        if (pos[i] < 0) {
          const long long x = mag_key((double)dq[i]);
          if (x > best) { best = x; bi = i; }
        }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        of->value = bi < n ? (double)dq[bi] : -1.0;
        of->own = bi < n ? (double)oq[bi] : 0.0;
        of->col = bi < n ? c0 + bi : n;
        sh_best = bi;
      }
    }
    __syncthreads();
    if (sh_best < n)
      for (int l = tid; l < j; l += kFacThreads) ofu[l] = U[l * w + sh_best];
    cta_sync(ct);
    // the winner of the cluster
    if (tid < 32) {
      const unsigned a = cluster_addr(of, lane < ct.size ? lane : ct.rank);
      const double v = lane < ct.size ? cluster_ld<double>(a) : -1.0;
      const double own = cluster_ld<double>(a + (unsigned)offsetof(Pivot, own));
      const int col = lane < ct.size ? cluster_ld<int>(a + (unsigned)offsetof(Pivot, col)) : n;
      long long best = mag_key(v);
      int bi = col, bl = lane;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o), ol = __shfl_xor_sync(0xffffffffu, bl, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; bl = ol; }
      }
      bl = __shfl_sync(0xffffffffu, bl, 0);
      if (lane == bl) {
        sh_win.value = v;
        sh_win.own = own;
        sh_win.col = col;
        sh_from = lane;
        sh_rs = R(1) / sqrt((R)v);
      }
    }
    __syncthreads();
    const double dp = sh_win.value, op = sh_win.own;
    const int p = sh_win.col, from = sh_from;
    if (j == 0) d0 = dp;
    if (p >= n || !(dp > rel * d0) || !(dp > 0.0)) return j;
    if (safe >= 0.0 && !(dp >= safe * op)) return -1;
    const R rs = sh_rs;
    R a_pc = R(0);
    if (tid < nl) a_pc = (R)A[(long long)p * lda + c0 + tid];
    {
      const unsigned a = cluster_addr(ofu, from);
      for (int l = tid; l < j; l += kFacThreads) uc[l] = cluster_ld<R>(a + (unsigned)(l * sizeof(R)));
    }
    if (tid == 0) perm[j] = p;
    __syncthreads();
    for (int e = tid; e < kFacSlices * nl; e += kFacThreads) {
      const int sl = e / nl, c = e - sl * nl;
      R acc = R(0);
#pragma unroll 8
      for (int l = sl; l < j; l += kFacSlices) acc = fma(uc[l], U[l * w + c], acc);
      part[e] = acc;
    }
    __syncthreads();
    if (tid < nl) {
      if (c0 + tid == p) {
        U[j * w + tid] = dq[tid] * rs;
        pos[tid] = j;
      } else if (pos[tid] < 0) {
        R acc = a_pc;
#pragma unroll
        for (int k = 0; k < kFacSlices; ++k) acc -= part[k * nl + tid];
        acc *= rs;
        U[j * w + tid] = acc;
        dq[tid] = fma(-acc, acc, dq[tid]);
      }
    }
    __syncthreads();
  }
  return n;
}

// Column-pivoted Householder QR of the M x r matrix B (leading dimension ld)
// in place: R in the upper trapezoid, the position order in perm; returns the
// rank.  Bound: the FP64 units, a quarter of the SM each (a warp operation holds one
// for 64 clocks).  Four warps, one per quarter, share the rows of 32 columns, so
// that only four partial sums a column are left to add, on every lane that needs
// them; sixteen row groups spent more on those sums than on the products.
// Class, 16 row groups -> four: 3x3 chi = 8 evolution 4.3 -> 3.5 ms, 4x4 chi = 12
// layer 2.4 -> 1.9.
__device__ int qrcp(double* B, int ld, int M, int r, double* dg, double* w, double* v, double* part, int* perm,
                    double rel) {
  __shared__ long long rv[32];
  __shared__ int ri[32];
  __shared__ double red[32];
  __shared__ double sh_h[3];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int CB = 32 * (kFacThreads / 128);              // columns of a pass
  const int rg = wid & 3, cb = 32 * (wid >> 2) + lane;      // row group, column of a pass
  for (int i = threadIdx.x; i < r; i += blockDim.x) perm[i] = i;
  for (int k = cb; k < r; k += CB) {
    double s = 0.0;
    for (int i = rg; i < M; i += 4) { const double x = B[(long long)i * ld + k]; s = fma(x, x, s); }
    part[rg * r + k] = s;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < r; k += blockDim.x) {
    const double s = (part[k] + part[r + k]) + (part[2 * r + k] + part[3 * r + k]);
    dg[k] = s;
    w[k] = s;   // reference norms for the downdate safeguard
  }
  __syncthreads();
  double n0 = 0.0;
  const int kmax = M < r ? M : r;
  for (int j = 0; j < kmax; ++j) {
    const int p = block_argmax(dg, j, r, rv, ri);
    const double dp = dg[p];
    if (j == 0) n0 = dp;
    if (!(dp > rel * rel * n0) || !(dp > 0.0)) return j;
    if (p != j) {
      for (int i = threadIdx.x; i < M; i += blockDim.x) {
        const double t = B[(long long)i * ld + j];
        B[(long long)i * ld + j] = B[(long long)i * ld + p];
        B[(long long)i * ld + p] = t;
      }
      if (threadIdx.x == 0) {
        const int t = perm[j]; perm[j] = perm[p]; perm[p] = t;
        double td = dg[j]; dg[j] = dg[p]; dg[p] = td;
        td = w[j]; w[j] = w[p]; w[p] = td;
      }
      __syncthreads();
    }
    if (wid < 4) {
      double s = 0.0;
      for (int i = j + threadIdx.x; i < M; i += 128) {
        const double x = B[(long long)i * ld + j];
        s = fma(x, x, s);
      }
      s = warp_sum(s);
      if (lane == 0) red[wid] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      reflector(B[(long long)j * ld + j], (red[0] + red[1]) + (red[2] + red[3]), sh_h[0], sh_h[2], sh_h[1]);
    __syncthreads();
    const double beta = sh_h[0], inv = sh_h[1], tau = sh_h[2];
    for (int i = j + threadIdx.x; i < M; i += blockDim.x) v[i] = (i == j) ? 1.0 : B[(long long)i * ld + j] * inv;
    __syncthreads();
    for (int i = j + threadIdx.x; i < M; i += blockDim.x) B[(long long)i * ld + j] = (i == j) ? beta : 0.0;
    for (int k = j + 1 + cb; k < r; k += CB) {
      double acc = 0.0;
      for (int i = j + rg; i < M; i += 4) acc = fma(v[i], B[(long long)i * ld + k], acc);
      part[rg * r + k] = acc;
    }
    __syncthreads();
    for (int k = j + 1 + cb; k < r; k += CB) {
      const double tw = tau * ((part[k] + part[r + k]) + (part[2 * r + k] + part[3 * r + k]));
      for (int i = j + rg; i < M; i += 4) B[(long long)i * ld + k] -= v[i] * tw;
    }
    __syncthreads();
    for (int k = j + 1 + threadIdx.x; k < r; k += blockDim.x) {
      const double rjk = B[(long long)j * ld + k];
      double nd = dg[k] - rjk * rjk;
      if (nd < 0.05 * w[k]) {  // cancellation: recompute the trailing norm
        nd = 0.0;
        for (int i = j + 1; i < M; ++i) { const double x = B[(long long)i * ld + k]; nd = fma(x, x, nd); }
        w[k] = nd;
      }
      dg[k] = nd;
    }
    __syncthreads();
  }
  return kmax;
}

// From a Gram (the Cholesky-QR branch; FP32 storage: every site): pivoted
// Cholesky of G (r x r, formed by k_form behind T).
// From a Householder R (FP64 storage): column-pivoted Householder QR of B (4k x r, in T).
// Output: T (rank x r upper trapezoidal, pivoted column order), perm[q] =
// original column of pivoted column q, rank -> ival.
//
// Whether the Cholesky-QR branch can be trusted with its Gram C = cv^T cv
// (n x n): its factor is only as accurate as C.  The Gram's rounding is
// relative to the norms of the columns it pairs (runs of 256 terms in FP32:
// ~1e-8 of that scale; FP64: ~1e-14), so a column that is a linear
// combination of the others in exact arithmetic keeps a Schur complement of
// that relative size, and the Q-less update would take the noise for a
// direction (Q = cv R^-1 is then far from orthonormal).  The pivoted Cholesky
// of C (in FP32 for FP32 storage) therefore checks every accepted pivot
// against the column's own diagonal; when one keeps less than rel_safe of it
// the site is marked branch 2 and left for the pass that follows (only = 2
// runs that pass only).  Pivots below rel of the first end the check
// (directions too small to matter: the factorisation of G cuts them as rank;
// rel_exact where G comes from an exact Gram).
//
// Measured, factor class of one saturated layer, right-looking Cholesky and one
// thread per column -> left-looking on a cluster, no Householder in FP32 storage: 4x4
// chi = 48 212 -> 6.3 ms, 3x3 chi = 100 357 -> 19 ms, 3x5 chi = 27 42 -> 2.1 ms.
__global__ void __launch_bounds__(kFacThreads)
k_factor(const SiteFacItem* __restrict__ items, int* ival, int only, unsigned long long* qcount, int rmax, int nmax,
         int householder, int csize) {
  const SiteFacItem it = items[blockIdx.x / csize];
  const int branch = ival[it.branch_idx];
  if (only >= 0 && branch != only) return;
  Cta ct;
  ct.rank = blockIdx.x % csize;
  ct.size = csize;
  ct.tid = (long long)ct.rank * blockDim.x + threadIdx.x;
  ct.nthr = (long long)csize * blockDim.x;
  if (qcount && ct.tid == 0 && branch == 0) atomicAdd(&qcount[0], 1ull);
  long long m;
  int n;
  cv_shape(it.cv, ival, m, n);
  const int chic = n / 4;
  const int rg = ival[it.rg_idx];
  const int r = rg * chic;
  double* T = it.T;
  const int ld = it.ldt;
  extern __shared__ __align__(16) unsigned char fsh[];
  __shared__ Pivot offer[2];
  const FacSmem S = fac_smem(rmax, nmax, householder, csize);
  const int ldo = rmax > nmax ? rmax : nmax;
  double* mat = reinterpret_cast<double*>(fsh + S.mat);
  int* pos = reinterpret_cast<int*>(fsh + S.pos);
  int* perm = reinterpret_cast<int*>(fsh + S.perm);
  const size_t room = S.total - S.mat;
  auto chol = [&](auto* zero, const double* A, int lda, int k, auto* scratch, double rel, double safe, auto*& U) -> int {
    using R = std::remove_reference_t<decltype(*zero)>;
    const int w = (k + csize - 1) / csize;
    U = sizeof(R) * (size_t)k * w <= room ? reinterpret_cast<R*>(mat) : scratch + (long long)ct.rank * w * k;
    return chol_cluster<R>(A, lda, k, w, U, ct, offer, reinterpret_cast<R*>(fsh + S.cand), ldo,
                           reinterpret_cast<R*>(fsh + S.uc), reinterpret_cast<R*>(fsh + S.part),
                           reinterpret_cast<R*>(fsh + S.dq), reinterpret_cast<R*>(fsh + S.oq), pos, perm, rel, safe);
  };
  double* scratch = T + (long long)2 * ld * ld;      // behind T and G: 2 ld^2 doubles
  if (branch == 1) {
    int ok;
    if (it.rel_safe >= 1e-6) {
      float* U;
      ok = chol((float*)nullptr, it.C, it.ldc, n, reinterpret_cast<float*>(scratch), it.rel, it.rel_safe, U);
    } else {
      double* U;
      ok = chol((double*)nullptr, it.C, it.ldc, n, scratch, it.rel, it.rel_safe, U);
    }
    if (ct.tid == 0 && qcount) atomicAdd(&qcount[ok >= 0 ? 1 : 2], 1ull);
    cta_sync(ct);                                    // the last offers are read, every CTA has its branch
    if (ok < 0) {
      if (ct.tid == 0) ival[it.branch_idx] = 2;
      return;
    }
  }
  if (branch == 1 || !householder) {
    double* U;
    const int rank = chol((double*)nullptr, T + (long long)ld * ld, ld, r, scratch, branch == 1 ? it.rel : it.rel_exact, -1.0, U);
    // columns that never became a pivot follow in their own order
    const int w = (r + csize - 1) / csize, c0 = ct.rank * w;
    const int nl = min(w, r - c0);
    int* taken = reinterpret_cast<int*>(fsh + S.uc);
    __syncthreads();
    for (int i = threadIdx.x; i < r; i += blockDim.x) taken[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < rank; i += blockDim.x) taken[perm[i]] = 1;
    __syncthreads();
    for (int c = threadIdx.x; c < nl; c += blockDim.x) {
      int q = pos[c];
      if (q < 0) {
        q = rank;
        for (int i = 0; i < c0 + c; ++i) q += 1 - taken[i];
        pos[c] = q;
      }
      it.perm[q] = c0 + c;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < rank * nl; e += blockDim.x) {
      const int a = e / nl, c = e - a * nl, q = pos[c];
      if (a <= q) T[(long long)a * ld + q] = U[a * w + c];
    }
    if (ct.tid == 0) ival[it.rank_idx] = rank;
    cta_sync(ct);                                    // no CTA leaves while its offers may be read
    return;
  }
  const int M = 4 * ival[it.kfac_idx];
  double* v = reinterpret_cast<double*>(fsh + S.v);
  double* part = v + (size_t)4 * nmax;
  double* dg = reinterpret_cast<double*>(fsh + S.dq);
  double* od = reinterpret_cast<double*>(fsh + S.oq);
  const bool in = sizeof(double) * (size_t)M * r <= room;
  if (in) {
    for (long long e = threadIdx.x; e < (long long)M * r; e += blockDim.x) {
      const int a = (int)(e / r), q = (int)(e - (long long)a * r);
      mat[e] = T[(long long)a * ld + q];
    }
    __syncthreads();
  }
  const int rank = qrcp(in ? mat : T, in ? r : ld, M, r, dg, od, v, part, perm, it.rel);
  __syncthreads();
  if (in)
    for (long long e = threadIdx.x; e < (long long)rank * r; e += blockDim.x) {
      const int a = (int)(e / r), q = (int)(e - (long long)a * r);
      T[(long long)a * ld + q] = mat[e];
    }
  for (int i = threadIdx.x; i < r; i += blockDim.x) it.perm[i] = perm[i];
  if (threadIdx.x == 0) ival[it.rank_idx] = rank;
}

cudaError_t launch_factor(const SiteFacItem* items, int n_items, int rmax, int nmax, int* ival,
                          cudaStream_t s, int only, int householder, unsigned long long* qcount) {
  if (n_items == 0) return cudaSuccess;
  // FP32 storage: up to eight CTAs a site while they all find an SM (a factor of
  // r = 4 chi columns below 128 is latency-bound on one); the Householder QR of
  // FP64 storage is one block's
  int csize = 1;
  if (!householder && rmax > 128)
    for (csize = 8; csize > 1 && n_items * csize > 2 * 152; csize /= 2) {}
  const FacSmem S = fac_smem(rmax, nmax, householder, csize);
  cudaError_t e = cudaFuncSetAttribute(k_factor, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S.total);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_items * csize);
  cfg.blockDim = dim3(kFacThreads);
  cfg.dynamicSmemBytes = S.total;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = csize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, k_factor, items, ival, only, qcount, rmax, nmax, householder, csize);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// ===================================================================== core
// Rotation of a Jacobi pair from its squared norms and product: h = tan(theta / 2) and
// s = sin theta of the smaller angle that makes the columns orthogonal, and the new
// squared norms.  False when the pair is orthogonal to tol (tol2 = tol^2),
// numerically zero or coupled by less than cut.
//
// The rotation is applied as x -= s (y + h x), y += s (x - h y) (the old x): four
// multiply-adds like the c, s form, but what rounding does to the columns' norms
// and angles scales with s, so the thousands of small late rotations leave V
// more orthogonal.  h may be off by 1e-7 of itself (the next sweep sees what that
// leaves); s has to belong to h.
__device__ __forceinline__ bool rot_params(float al, float be, float ga, float tol2, float negligible, float cut, float& h,
                                           float& s, float& na, float& nb) {
  if (!(ga != 0.f && al > negligible && be > negligible && fabsf(ga) > cut &&
        fabsf(ga) * rsqrtf(al) * rsqrtf(be) * fabsf(ga) * rsqrtf(al) * rsqrtf(be) > tol2))
    return false;
  const float z = __fdividef(be - al, 2.f * ga), az = fabsf(z);
  const float t = copysignf(az > 1e8f ? 0.5f / az : __fdividef(1.f, az + sqrtf(fmaf(z, z, 1.f))), z);
  h = __fdividef(t, 1.f + sqrtf(fmaf(t, t, 1.f)));
  s = 2.f * h / fmaf(h, h, 1.f);
  na = al - t * ga;
  nb = be + t * ga;
  return true;
}
// FP64: an operation of a warp holds its quarter of the FP64 unit for 64 clocks
// (measured; independent ones are no faster), so what need not be FP64 is not.
// The test and h come from the operands' leading 24 bits, scaled to the largest
// (integer work); s = 2 h / (1 + h^2) follows from an FP32 reciprocal by one
// cubic step, 2 h times it being exact; the norms' updates take tan theta in FP32
// (they steer the next rotations and are recomputed every round).
__device__ __forceinline__ bool rot_params(double al, double be, double ga, double tol2, double negligible, double cut,
                                           double& h, double& s, double& na, double& nb) {
  // al, be, |ga| and the bounds are not negative: their bits order like their values
  const long long ia = __double_as_longlong(al), ib = __double_as_longlong(be);
  const long long ig = __double_as_longlong(ga) & 0x7fffffffffffffffll;
  const int e = (int)(max(max(ia, ib), ig) >> 52);
  if (e >= 0x7ff || ig == 0 || min(ia, ib) <= __double_as_longlong(negligible) || ig <= __double_as_longlong(cut)) return false;
  const float fa = top_float(al, e), fb = top_float(be, e), fg = top_float(ga, e);
  const float rel = fabsf(fg) * rsqrtf(fa) * rsqrtf(fb);
  if (!(rel * rel > (float)tol2)) return false;
  const double d = be - al;
  const float df = top_float(d, e), z = __fdividef(df, 2.f * fg), az = fabsf(z);
  const float t = copysignf(az > 1e8f ? 0.5f / az : 1.f / (az + sqrtf(fmaf(z, z, 1.f))), z);
  const float hf = t / (1.f + sqrtf(fmaf(t, t, 1.f)));
  if (!(fabsf(hf) > 1e-30f)) return false;                      // beyond FP32's range: no rotation either
  h = wide(hf);
  const double y = wide(__frcp_rn(fmaf(hf, hf, 1.f)));
  const double r = fma(-fma(h, h, 1.0), y, 1.0);
  const double w = wide(2.f * hf) * y;
  s = fma(w, fma(r, r, r), w);
  const double tg = wide(t) * ga;
  na = al - tg;
  nb = be + tg;
  return true;
}
__device__ __forceinline__ void rot_apply(float& x, float& y, float h, float s) {
  const float u = fmaf(h, x, y), v = fmaf(-h, y, x);
  x = fmaf(-s, u, x);
  y = fmaf(s, v, y);
}
// the same rotation as three shears: three FP64 operations a pair instead of four
__device__ __forceinline__ void rot_apply(double& x, double& y, double h, double s) {
  x = fma(-h, y, x);
  y = fma(s, x, y);
  x = fma(-h, y, x);
}

// Pair pi of a round of the tournament of n columns (np = n rounded up to even);
// x < 0: the one with the dummy.
__device__ __forceinline__ int2 tournament(int round, int pi, int n, int np) {
  int a, b;
  if (pi == 0) { a = np - 1; b = round; }
  else {
    a = round + pi; if (a >= np - 1) a -= np - 1;
    b = round - pi; if (b < 0) b += np - 1;
  }
  if (a >= n || b >= n) return make_int2(-1, -1);
  return a < b ? make_int2(a, b) : make_int2(b, a);
}

// One-sided Jacobi (Hestenes) on the columns of A (n x n, column-major, leading
// dimension ld), accumulating V (the same), by one block.  Returns the
// sweep count; sets *capped when the sweep budget ran out.
//
// A pair of columns belongs to L lanes that hold E values of both in registers
// from the dot product to the rotation (V's too, requested before the product is
// summed, where the registers hold them: up to four values a lane); the squared norms are recomputed every sweep and updated by the
// rotations between, so a pair costs one reduction.  Bound: the instructions of
// a round (the scalars of a rotation are ~80 and repeat per warp, so a warp takes
// 32 / L pairs) and its latency, then shared-memory bandwidth.  ld is L more
// than a multiple of 32, so that the L-lane groups of a warp, whose columns are
// neighbours, read different banks.  FP64 goes this way up to n = 16 (the pairs'
// warps then have a quarter of the FP64 unit each; one barrier a round).
__host__ __device__ inline int jac_lanes(int n) { return n <= 32 ? 8 : 16; }
__host__ __device__ inline int jac_ld(int n) {
  const int L = jac_lanes(n);
  return n <= L ? L : (n - L + 31) / 32 * 32 + L;
}
template <typename R, int L, int E>
__device__ int jacobi_block_l(R* A, int n, int ld, R* V, R* nrm, int max_sweeps, int* capped) {
  const int l = threadIdx.x % L, grp = threadIdx.x / L, ng = blockDim.x / L;
  const unsigned mask = (L == 16 ? 0xffffu : 0xffu) << (threadIdx.x & 31 & ~(L - 1));
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) V[e / n * ld + e % n] = e % (n + 1) == 0 ? R(1) : R(0);
  auto norms = [&]() {
    for (int c = grp; c < n; c += ng) {
      R q = 0;
#pragma unroll
      for (int u = 0; u < E; ++u) {
        const int i = l + L * u;
        if (i < n) q = fma(A[c * ld + i], A[c * ld + i], q);
      }
#pragma unroll
      for (int o = L / 2; o > 0; o >>= 1) q += __shfl_xor_sync(mask, q, o);
      if (l == 0) nrm[c] = q;
    }
    __syncthreads();
  };
  norms();
  if (n < 2) return 0;
  // ||A||_F^2 (the same bits whatever the block's size)
  R fro = 0;
  for (int c = threadIdx.x & 31; c < n; c += 32) fro += nrm[c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, o);
  __syncthreads();
  const int np = (n % 2) ? n + 1 : n;   // players incl. a dummy
  // orthogonality target: above the rounding noise of a length-n dot product in
  // the working precision (FP32 columns: ~sqrt(n) 6e-8 relative); columns below
  // 1e-30 (FP64) or 1e-13 (FP32) of the total squared norm are numerically zero:
  // rotating them only stirs rounding noise and never converges
  const double tol = (sizeof(R) == 4 ? 3e-7 : 1e-15) * sqrt((double)n);
  const R tol2 = (R)(tol * tol);
  const R negligible = (R)(sizeof(R) == 4 ? 1e-13 : 1e-30) * fro;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (sweep > 0) norms();
    int rotated = 0;
    for (int round = 0; round < np - 1; ++round) {
      for (int pi = grp; pi < np / 2; pi += ng) {
        const int2 pq = tournament(round, pi, n, np);
        if (pq.x < 0) continue;
        R* Ap = A + pq.x * ld + l;
        R* Aq = A + pq.y * ld + l;
        R* Vp = V + pq.x * ld + l;
        R* Vq = V + pq.y * ld + l;
        R x[E], y[E], vx[E], vy[E], ga = 0;
#pragma unroll
        for (int u = 0; u < E; ++u) {
          const bool in = l + L * u < n;
          x[u] = in ? Ap[L * u] : R(0);
          y[u] = in ? Aq[L * u] : R(0);
          if (E <= 4) {
            vx[u] = in ? Vp[L * u] : R(0);
            vy[u] = in ? Vq[L * u] : R(0);
          }
        }
        const R al = nrm[pq.x], be = nrm[pq.y];
#pragma unroll
        for (int u = 0; u < E; ++u) ga = fma(x[u], y[u], ga);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) ga += __shfl_xor_sync(mask, ga, o);
        R h, s, na, nb;
        if (rot_params(al, be, ga, tol2, negligible, R(0), h, s, na, nb)) {
          rotated = 1;
#pragma unroll
          for (int u = 0; u < E; ++u) {
            if (l + L * u < n) {
              if (E > 4) {
                vx[u] = Vp[L * u];
                vy[u] = Vq[L * u];
              }
              rot_apply(x[u], y[u], h, s);
              rot_apply(vx[u], vy[u], h, s);
              Ap[L * u] = x[u];
              Aq[L * u] = y[u];
              Vp[L * u] = vx[u];
              Vq[L * u] = vy[u];
            }
          }
          if (l == 0) { nrm[pq.x] = na; nrm[pq.y] = nb; }
        }
      }
      __syncthreads();
    }
    if (!__syncthreads_or(rotated)) break;
  }
  if (sweep >= max_sweeps && threadIdx.x == 0) *capped = 1;
  __syncthreads();
  return sweep;
}

constexpr int kCoreThreads = 512;                  // 128 registers: columns stay in them
constexpr size_t kCoreSmem = (size_t)192 * 1024;
constexpr int kCoreMaxDim = 512;                   // columns and rows of a core: rg * chi <= 512

// Column of up to 32 U values, 32 apart per lane (zeros past len).
template <int U>
__device__ __forceinline__ void col_load(float (&a)[U], const float* x, int len) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = (threadIdx.x & 31) + 32 * u;
    a[u] = i < len ? x[i] : 0.f;
  }
}
template <int U>
__device__ __forceinline__ void col_store(const float (&a)[U], float* x, int len) {
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = (threadIdx.x & 31) + 32 * u;
    if (i < len) x[i] = a[u];
  }
}
template <int U>
__device__ __forceinline__ float col_dot(const float (&a)[U], const float (&b)[U]) {
  float ga = 0;
#pragma unroll
  for (int u = 0; u < U; ++u) ga = fmaf(a[u], b[u], ga);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
  return ga;
}

// One warp's FP32 rotation of the columns x and y (length m, shared memory) of A
// and vx, vy (length nv) of V; nx, ny are their squared norms, kept up to date.
// Returns whether it rotated.  m and nv are at most 32 U.
template <int U>
__device__ __noinline__ int jac_pair(float* x, float* y, int m, float* vx, float* vy, int nv, float* nx, float* ny,
                                     float tol2, float negligible, float cut) {
  float a[U], b[U];
  col_load(a, x, m);
  col_load(b, y, m);
  float h, s, na, nb;
  if (!rot_params(*nx, *ny, col_dot(a, b), tol2, negligible, cut, h, s, na, nb)) return 0;
#pragma unroll
  for (int u = 0; u < U; ++u) rot_apply(a[u], b[u], h, s);
  col_store(a, x, m);
  col_store(b, y, m);
  col_load(a, vx, nv);
  col_load(b, vy, nv);
#pragma unroll
  for (int u = 0; u < U; ++u) rot_apply(a[u], b[u], h, s);
  col_store(a, vx, nv);
  col_store(b, vy, nv);
  __syncwarp();
  if ((threadIdx.x & 31) == 0) { *nx = na; *ny = nb; }
  return 1;
}

// The cross pairs of two blocks of columns in shared memory (cp columns at slot
// 0, then cq; per values each: m of A, nv of V): step k pairs column i of the first
// with column (i + k) mod bs of the second.  Bound: the latency of a step (load,
// product, rotation, store, barrier), then shared-memory bandwidth.  So a warp
// keeps its column of the first block in registers over all steps and moves only
// the other one.  Up to 256 rows it holds A's and V's; above that (up to 32
// columns a block: two per warp) the rotations are kept and V follows in a
// pass of its own.  hs: (h, s) of step k and column i at 32 k + i, s = 2: none.
template <int U>
__device__ __noinline__ int jac_cross(float* buf, int per, int m, int nv, int cp, int cq, int bs, float* nrm,
                                      float tol2, float negligible, float cut, float2* hs) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  constexpr int NW = kCoreThreads / 32;
  int rot = 0;
  if constexpr (U <= 8) {                                   // 32 U >= n: bs <= 16 = NW
    const int i = wid;
    const bool on = i < cp;
    float* xc = buf + i * per;
    float x[U], vx[U], nx = 0.f;
    if (on) {
      col_load(x, xc, m);
      col_load(vx, xc + m, nv);
      nx = nrm[i];
    }
    int q = i;                                              // (i + k) mod bs
    for (int k = 0; k < bs; ++k) {
      if (on && q < cq) {
        float* yc = buf + (cp + q) * per;
        float* ny = nrm + cp + q;
        float y[U], vy[U], h, s, na, nb;
        col_load(y, yc, m);
        col_load(vy, yc + m, nv);
        if (rot_params(nx, *ny, col_dot(x, y), tol2, negligible, cut, h, s, na, nb)) {
          rot = 1;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            rot_apply(x[u], y[u], h, s);
            rot_apply(vx[u], vy[u], h, s);
          }
          col_store(y, yc, m);
          col_store(vy, yc + m, nv);
          nx = na;
          __syncwarp();
          if (lane == 0) *ny = nb;
        }
      }
      if (++q >= bs) q = 0;
      __syncthreads();
    }
    if (on) {
      col_store(x, xc, m);
      col_store(vx, xc + m, nv);
    }
  } else {
    float x[2][U], nx[2];
    int q[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = wid + NW * c;
      q[c] = i;
      col_load(x[c], buf + i * per, i < cp ? m : 0);
      nx[c] = i < cp ? nrm[i] : 0.f;
    }
    for (int k = 0; k < bs; ++k) {
      float y[2][U], ga[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) col_load(y[c], buf + (cp + q[c]) * per, wid + NW * c < cp && q[c] < cq ? m : 0);
#pragma unroll
      for (int c = 0; c < 2; ++c) ga[c] = col_dot(x[c], y[c]);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int i = wid + NW * c;
        if (i < cp && q[c] < cq) {
          float* ny = nrm + cp + q[c];
          float2 r;
          float na, nb;
          if (rot_params(nx[c], *ny, ga[c], tol2, negligible, cut, r.x, r.y, na, nb)) {
            rot = 1;
#pragma unroll
            for (int u = 0; u < U; ++u) rot_apply(x[c][u], y[c][u], r.x, r.y);
            col_store(y[c], buf + (cp + q[c]) * per, m);
            nx[c] = na;
            __syncwarp();
            if (lane == 0) *ny = nb;
          } else {
            r.y = 2.f;
          }
          if (lane == 0) hs[32 * k + i] = r;
        }
        if (++q[c] >= bs) q[c] -= bs;
      }
      __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = wid + NW * c;
      if (i < cp) col_store(x[c], buf + i * per, m);
      q[c] = i;
      col_load(x[c], buf + i * per + m, i < cp ? nv : 0);
    }
    for (int k = 0; k < bs; ++k) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int i = wid + NW * c;
        if (i < cp && q[c] < cq) {
          const float2 r = hs[32 * k + i];
          if (r.y < 1.5f) {
            float y[U];
            float* yc = buf + (cp + q[c]) * per + m;
            col_load(y, yc, nv);
#pragma unroll
            for (int u = 0; u < U; ++u) rot_apply(x[c][u], y[u], r.x, r.y);
            col_store(y, yc, nv);
          }
        }
        if (++q[c] >= bs) q[c] -= bs;
      }
      __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int i = wid + NW * c;
      if (i < cp) col_store(x[c], buf + i * per + m, nv);
    }
  }
  __syncthreads();
  return rot;
}

// The pairs f(0) .. f(cnt - 1) of one inner round in FP64 (the columns .x and .y of
// buf, x < 0: none; per values each, m of A then nv of V), by the whole block: half
// a warp per dot product (a warp above 64 rows), one lane per pair for the
// rotation, a warp per 32 rows of a pair to rotate.  Bound: the FP64 units, one
// warp operation per 64 clocks and quarter of the SM: an operation that all lanes
// repeat costs as much as 32 useful ones, and the quarters share the work by
// warps.
struct JacRound {
  double ga[64], h[64], s[64];                             // s > 1.5: no rotation
};
template <class F>
__device__ __forceinline__ int jac_round64(JacRound& R, int cnt, F f, double* buf, int per, int m, int nv, double* nrm,
                                           double tol2, double negligible, double cut) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int rot = 0;
  if (m > 64) {
    for (int k = wid; k < cnt; k += nw) {
      const int2 v = f(k);
      if (v.x < 0) continue;
      const double* x = buf + v.x * per;
      const double* y = buf + v.y * per;
      double ga = 0.0;
      for (int i = lane; i < m; i += 32) ga = fma(x[i], y[i], ga);
      ga = warp_sum(ga);
      if (lane == 0) R.ga[k] = ga;
    }
  } else {
    const int l = threadIdx.x & 15;
    const unsigned mask = 0xffffu << (threadIdx.x & 16);
    for (int k = threadIdx.x >> 4; k < cnt; k += 2 * nw) {
      const int2 v = f(k);
      if (v.x < 0) continue;
      const double* x = buf + v.x * per;
      const double* y = buf + v.y * per;
      double ga = 0.0;
      for (int i = l; i < m; i += 16) ga = fma(x[i], y[i], ga);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) ga += __shfl_xor_sync(mask, ga, o);
      if (l == 0) R.ga[k] = ga;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < cnt; k += blockDim.x) {
    const int2 v = f(k);
    double h = 0.0, s = 2.0, na, nb;
    if (v.x >= 0 && rot_params(nrm[v.x], nrm[v.y], R.ga[k], tol2, negligible, cut, h, s, na, nb)) {
      nrm[v.x] = na;
      nrm[v.y] = nb;
      rot = 1;
    }
    R.h[k] = h;
    R.s[k] = s;
  }
  __syncthreads();
  const int segs = (m + nv + 31) >> 5;
  for (int e = wid; e < cnt * segs; e += nw) {
    const int k = e / segs, i = 32 * (e - k * segs) + lane;
    const double s = R.s[k];
    if (s > 1.5) continue;
    const int2 v = f(k);
    if (i < m + nv) {
      double* x = buf + v.x * per + i;
      double* y = buf + v.y * per + i;
      double p = *x, q = *y;
      rot_apply(p, q, R.h[k], s);
      *x = p;
      *y = q;
    }
  }
  __syncthreads();
  return rot;
}

// The same in FP64, in rounds of jac_round64.  buf: columns of 2 n values, A's then V's
// (A filled in by the caller).
__device__ int jacobi_block64(double* buf, int n, double* nrm, int max_sweeps, int* capped, JacRound& R) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int per = 2 * n, np = n + (n & 1);
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) buf[e / n * per + n + e % n] = e % (n + 1) == 0 ? 1.0 : 0.0;
  auto norms = [&]() {
    for (int c = wid; c < n; c += nw) {
      double q = 0.0;
      for (int i = lane; i < n; i += 32) q = fma(buf[c * per + i], buf[c * per + i], q);
      q = warp_sum(q);
      if (lane == 0) nrm[c] = q;
    }
    __syncthreads();
  };
  norms();
  if (n < 2) return 0;
  double fro = 0.0;
  for (int c = lane; c < n; c += 32) fro += nrm[c];
  fro = warp_sum(fro);
  __syncthreads();
  const double tol = 1e-15 * sqrt((double)n), negligible = 1e-30 * fro;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (sweep > 0) norms();
    int rotated = 0;
    for (int round = 0; round < np - 1; ++round)
      rotated |= jac_round64(R, np / 2, [&](int pi) { return tournament(round, pi, n, np); }, buf, per, n, n, nrm,
                             tol * tol, negligible, 0.0);
    if (!__syncthreads_or(rotated)) break;
  }
  if (sweep >= max_sweeps && threadIdx.x == 0) *capped = 1;
  __syncthreads();
  return sweep;
}

// One-sided Jacobi of A (m x n, column-major, leading dimension m, global
// memory) with the rotations accumulated in V (n x n), on all CTAs of the
// cluster.  The columns are cut into (at most) 16 blocks; a round of the block
// tournament pairs every block with another, and the columns of a pair of
// blocks meet each other in inner rounds of disjoint pairs, one warp per pair of
// columns (round 0: every pair within and across the two blocks; then the cross
// pairs only).  Each CTA brings its pairs of blocks into shared memory (A and V
// columns) and writes them back, so the matrix crosses L2 once per round of
// ~bs^2 rotations per CTA instead of twice per rotation; a matrix that one CTA
// holds stays there for all sweeps when the cluster is that CTA (a batch of
// many cores) or when there is too little to share (n <= 32: rank 0 works).
// The order of the rotations of a column depends on n alone, so every cluster
// size gives the same bits.
//
// Rotation and stopping rules as jacobi_block_l, plus abs_rel > 0: a pair whose
// coupling |a_p . a_q| is below abs_rel ||A||_F^2 is skipped too.  Such a pair
// moves no singular value by more than that, and without the cut the columns of
// tiny singular values (mostly rounding noise from rotations with the large
// ones) are chased for many sweeps without ever reaching relative
// orthogonality.  Squared norms are recomputed every round (up to n = 32 every
// sweep) and updated by the rotations between.  flags: 3 ints, zeroed by the
// caller; cnorm: n doubles.
template <typename R>
__device__ __noinline__ int jacobi_cluster(R* A, int m, int n, R* V, int max_sweeps, int* capped, double abs_rel, const Cta& ct,
                              int* flags, double* cnorm, unsigned char* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __shared__ double fr[32];
  // V = I and ||A||_F^2, by columns (its bits do not depend on the cluster)
  for (long long e = ct.tid; e < (long long)n * n; e += ct.nthr) V[e] = (e % (n + 1) == 0) ? R(1) : R(0);
  for (long long j = ct.tid >> 5; j < n; j += ct.nthr >> 5) {
    double q = 0.0;
    for (int i = lane; i < m; i += 32) { const double x = (double)A[j * m + i]; q = fma(x, x, q); }
    q = warp_sum(q);
    if (lane == 0) cnorm[j] = q;
  }
  cta_sync(ct);
  if (n < 2) return 0;
  double fro = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) fro += cnorm[j];
  fro = block_sum(fro, fr);
  const double tol = (sizeof(R) == 4 ? 3e-7 : 1e-15) * sqrt((double)m);
  const R tol2 = (R)(tol * tol);
  __shared__ union {
    JacRound jr;                                            // FP64
    float2 hs[32 * 32];                                     // FP32
  } rs;
  // columns below 1e-30 (FP64) or 1e-22 (FP32) of the total squared norm are
  // numerically zero: kept values reach 1e-11 of the largest, and the FP32 pass has
  // to find their directions too (a rotation keeps a small column's relative
  // accuracy; with 1e-13 the spectra of a 4x4, chi = 40 run were 3e-4 off after 19
  // steps, now 4e-7)
  const R negligible = (R)((sizeof(R) == 4 ? 1e-22 : 1e-30) * fro);
  const R abs_cut = (R)(abs_rel * fro);
  const int longest = max(m, n);                            // of a column: registers per lane
  const int room = (int)((kCoreSmem - 4096) / sizeof(R));
  R* nrm = reinterpret_cast<R*>(sh);                        // squared norms of the columns at hand
  R* buf = reinterpret_cast<R*>(sh + 4096);
  const int per = m + n;                                    // A column then V column
  int most = room / per / 2;                                // columns of a block: two blocks at a time
  if (most > 32) most = 32;
  int nblk = n < 16 ? n + (n & 1) : 16;
  if ((n + nblk - 1) / nblk > most) nblk = ((n + most - 1) / most + 1) / 2 * 2;
  const int bs = (n + nblk - 1) / nblk, npair = nblk / 2;
  const bool resident = (long long)per * n <= room && (ct.size == 1 || n <= 32);
  auto first = [&](int blk) { return min(blk * bs, n); };
  auto count = [&](int blk) { return min(bs, n - first(blk)); };
  // blocks P < Q of pair pi in a round
  auto blocks = [&](int round, int pi, int& P, int& Q) {
    if (pi == 0) { P = nblk - 1; Q = round; }
    else {
      P = round + pi; if (P >= nblk - 1) P -= nblk - 1;
      Q = round - pi; if (Q < 0) Q += nblk - 1;
    }
    if (P > Q) { const int t = P; P = Q; Q = t; }
  };
  auto col_sq = [&](const R* x) -> R {                      // squared norm of a column of A, by a warp
    R q = 0;
    for (int i = lane; i < m; i += 32) q = fma(x[i], x[i], q);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
    return q;
  };
  // columns c0 .. of the first cnt0 slots and d0 .. of the next cnt1 between global and
  // shared memory: a warp per column of A or V, eight values of a lane in flight; on the
  // way in, also the squared norms
  auto move = [&](bool in, int c0, int cnt0, int d0, int cnt1) {
    for (int t = wid; t < 2 * (cnt0 + cnt1); t += nw) {
      const int c = t >> 1;
      const long long col = c < cnt0 ? c0 + c : d0 + c - cnt0;
      R* g = (t & 1) ? V + col * n : A + col * m;
      R* l = buf + c * per + ((t & 1) ? m : 0);
      const int len = (t & 1) ? n : m;
      const R* src = in ? g : l;
      R* dst = in ? l : g;
      for (int i0 = lane; i0 < len; i0 += 256) {
        R v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (i0 + 32 * u < len) v[u] = src[i0 + 32 * u];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (i0 + 32 * u < len) dst[i0 + 32 * u] = v[u];
      }
      if (in && !(t & 1)) {
        __syncwarp();
        const R q = col_sq(l);
        if (lane == 0) nrm[c] = q;
      }
    }
    __syncthreads();
  };
  auto norms = [&](int cnt) {
    for (int c = wid; c < cnt; c += nw) {
      const R q = col_sq(buf + c * per);
      if (lane == 0) nrm[c] = q;
    }
    __syncthreads();
  };
  // the pairs f(0) .. f(cnt - 1) (slots of disjoint columns; x < 0: none), then a block barrier
  auto round_of = [&](int cnt, auto f) -> int {
    int rot = 0;
    if constexpr (sizeof(R) == 4) {
      for (int k = wid; k < cnt; k += nw) {
        const int2 v = f(k);
        if (v.x < 0) continue;
        R* x = buf + v.x * per;
        R* y = buf + v.y * per;
        R* nx = nrm + v.x;
        R* ny = nrm + v.y;
        if (longest <= 128) rot |= jac_pair<4>(x, y, m, x + m, y + m, n, nx, ny, tol2, negligible, abs_cut);
        else if (longest <= 256) rot |= jac_pair<8>(x, y, m, x + m, y + m, n, nx, ny, tol2, negligible, abs_cut);
        else rot |= jac_pair<16>(x, y, m, x + m, y + m, n, nx, ny, tol2, negligible, abs_cut);
      }
      __syncthreads();
    } else {
      rot = jac_round64(rs.jr, cnt, f, buf, per, m, n, nrm, tol2, negligible, abs_cut);
    }
    return rot;
  };
  // inner round `k` of block pair (P, Q) at slots p0, q0: pair i of it
  auto inner = [&](bool all, int k, int i, int P, int Q, int p0, int q0) -> int2 {
    const int cp = count(P), cq = count(Q);
    if (!all) {                                             // column i of P with column (i + k) mod bs of Q
      const int q = i + k < bs ? i + k : i + k - bs;
      return i < cp && q < cq ? make_int2(p0 + i, q0 + q) : make_int2(-1, -1);
    }
    const int cnt = cp + cq, np = cnt + (cnt & 1);          // tournament (a dummy if odd)
    if (k >= np - 1 || i >= np / 2) return make_int2(-1, -1);
    int x, y;
    if (i == 0) { x = np - 1; y = k; }
    else {
      x = k + i; if (x >= np - 1) x -= np - 1;
      y = k - i; if (y < 0) y += np - 1;
    }
    if (x >= cnt || y >= cnt) return make_int2(-1, -1);
    if (x > y) { const int t = x; x = y; y = t; }
    return make_int2(x < cp ? p0 + x : q0 + x - cp, y < cp ? p0 + y : q0 + y - cp);
  };
  const int steps0 = 2 * bs - 1;                            // inner rounds of round 0; later: bs
  int sweep = 0;
  if (resident && ct.rank == 0) move(true, 0, n, 0, 0);
  for (; sweep < max_sweeps; ++sweep) {
    int* flag = flags + sweep % 3;
    if (ct.rank == 0 && threadIdx.x == 0) flags[(sweep + 1) % 3] = 0;
    int rot = 0;
    for (int round = 0; round < nblk - 1; ++round) {
      const bool all = round == 0;
      const int steps = all ? steps0 : bs;
      if (resident) {
        if (ct.rank == 0) {
          // (up to n = 32 no cluster size takes the columns apart: once a sweep, as 15
          // times cost as much as the rotations)
          if (round == 0 || n > 32) norms(n);
          for (int k = 0; k < steps; ++k)
            rot |= round_of(npair * bs, [&](int e) {
              const int pi = e / bs, i = e - pi * bs;
              int P, Q;
              blocks(round, pi, P, Q);
              return inner(all, k, i, P, Q, first(P), first(Q));
            });
        }
      } else {
        for (int pi = ct.rank; pi < npair; pi += ct.size) {
          int P, Q;
          blocks(round, pi, P, Q);
          const int cp = count(P), cq = count(Q);
          if (cp == 0 || (cq == 0 && !all)) continue;
          move(true, first(P), cp, first(Q), cq);
          bool cross = false;
          if constexpr (sizeof(R) == 4) {
            cross = !all;
            if (cross) {
              if (longest <= 128) rot |= jac_cross<4>(buf, per, m, n, cp, cq, bs, nrm, tol2, negligible, abs_cut, rs.hs);
              else if (longest <= 256) rot |= jac_cross<8>(buf, per, m, n, cp, cq, bs, nrm, tol2, negligible, abs_cut, rs.hs);
              else rot |= jac_cross<16>(buf, per, m, n, cp, cq, bs, nrm, tol2, negligible, abs_cut, rs.hs);
            }
          }
          for (int k = 0; !cross && k < steps; ++k)
            rot |= round_of(bs, [&](int i) { return inner(all, k, i, P, Q, 0, cp); });
          move(false, first(P), cp, first(Q), cq);
        }
        cta_sync(ct);
      }
    }
    if (__syncthreads_or(rot) && threadIdx.x == 0) atomicOr(flag, 1);
    cta_sync(ct);
    if (*reinterpret_cast<volatile int*>(flag) == 0) break;
  }
  if (resident && ct.rank == 0) move(false, 0, n, 0, 0);
  if (sweep >= max_sweeps && threadIdx.x == 0) *capped = 1;
  cta_sync(ct);
  return sweep;
}

// Sign of a singular pair.  It is a gauge of the state that single-layer BP feels: it
// starts from the positive square roots of the messages' diagonals and stops at a
// tolerance, so signs left to rounding move C(t) by ~bp_tol^2 and may lead BP into
// another fixed point.  The sign is therefore a function of the state alone: of
// g_1 = X_1^T u and g_2 = X_2^T v (u, v the pair's vectors), which do not depend on
// the order of the pivots or on the signs of reflections.  (Where X_1 has full rank
// g_2 / sqrt(s) is the new index's column over the old ones, sqrt(s) X_1^+ u; where it
// has not, that column is not unique, but g_2 is.)
//
// A pair is turned the way in which the new index carries the old messages' positive
// vectors on the identity component: x = cos(m_1, g_2) + cos(m_2, g_1).  An index
// made by the odd Schmidt factors of the gate alone has no identity component and
// x is rounding noise; below kSignFloor the first entry of g_1 within 10 % of its
// largest is made positive instead.
//
// Entries are taken to FP32 by integer operations (FP64 conversions hold the FP64 unit
// for 64 clocks a warp); T is upper trapezoidal in the pivots' order.  A thread owns a
// column of T and up to eight pairs, so T is read once per eight pairs; the pairs are
// shared out over the cluster's CTAs.  Core class of a saturated layer, no rule (FP64)
// or one that read FP32 noise -> this one: 4x4 chi = 12 FP64 4.05 -> 4.11 ms, 4x4
// chi = 64 24.6 -> 24.5, 3x3 chi = 100 89.0 -> 90.1 (94 with a warp per pair, which reads
// T once per pair).
constexpr float kSignFloor = 1e-3f;
struct FactorSide {
  const double* T;         // k x r, leading dimension ld
  const int* perm;         // original column of each position
  int ld, k;
};
// vec(side, c): pair c's vector of that side times 2^(ex(side, c) - 1023) or less; m[side]:
// r values each.  Signs of this CTA's pairs -> out.  sh: kSignSmem floats.
constexpr int kSignPairs = 8;
constexpr int kSignSmem = 3 * kSignPairs * kCoreThreads;
template <class Vec, class Ex>
__device__ __noinline__ void pair_signs(const FactorSide s1, const FactorSide s2, int r, int chi, Vec vec, Ex ex,
                                        const float* m, const Cta& ct, double* out, float* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r32 = (r + 31) & ~31, ng = kCoreThreads / r32;   // r <= kCoreMaxDim = the threads
  const int grp = threadIdx.x / r32, q = threadIdx.x - grp * r32;
  float* us = sh;                                            // [group][row][pair of the group]
  float* gs = sh + kSignPairs * kCoreThreads;                // [side][pair][r32]
  const int per = (chi + ct.size - 1) / ct.size;
  const int end = min(chi, (ct.rank + 1) * per);
  for (int c0 = ct.rank * per; c0 < end; c0 += kSignPairs * ng) {
    const int n = min(kSignPairs * ng, end - c0);            // pair c0 + i: group i % ng, slot i / ng
    for (int side = 0; side < 2; ++side) {
      const FactorSide s = side == 0 ? s1 : s2;
      __syncthreads();
      for (int e = threadIdx.x; e < n * s.k; e += kCoreThreads) {
        const int i = e / s.k, a = e - i * s.k;
        us[((i % ng) * s.k + a) * kSignPairs + i / ng] = top_float(vec(side, c0 + i)[a], ex(side, c0 + i));
      }
      __syncthreads();
      if (grp < ng && grp < n) {
        const int et = s.k > 0 ? (__double2hiint(s.T[0]) >> 20) & 0x7ff : 0;   // the largest column's norm
        const int rows = min(s.k, (q | 31) + 1);
        const float4* u = reinterpret_cast<const float4*>(us + (size_t)grp * s.k * kSignPairs);
        float g[kSignPairs] = {};
#pragma unroll 8
        for (int a = 0; a < rows; ++a) {
          const float t = a <= q && q < r ? top_float(s.T[(long long)a * s.ld + q], et) : 0.f;
          const float4 x = u[2 * a], y = u[2 * a + 1];
          g[0] = fmaf(t, x.x, g[0]); g[1] = fmaf(t, x.y, g[1]); g[2] = fmaf(t, x.z, g[2]); g[3] = fmaf(t, x.w, g[3]);
          g[4] = fmaf(t, y.x, g[4]); g[5] = fmaf(t, y.y, g[5]); g[6] = fmaf(t, y.z, g[6]); g[7] = fmaf(t, y.w, g[7]);
        }
#pragma unroll
        for (int p = 0; p < kSignPairs; ++p)
          if (p * ng + grp < n) gs[(side * kSignPairs * ng + p * ng + grp) * r32 + q] = g[p];
      }
    }
    __syncthreads();
    for (int i = wid; i < n; i += kCoreThreads / 32) {
      float x = 0.f, turn = 1.f;
      for (int side = 0; side < 2; ++side) {
        const FactorSide s = side == 0 ? s1 : s2;
        const float* g = gs + (side * kSignPairs * ng + i) * r32;
        const float* w = m + (1 - side) * r;                 // m_2 meets g_1, m_1 meets g_2
        float d = 0.f, gg = 0.f, mm = 0.f, top = 0.f;
        for (int j = lane; j < r; j += 32) {
          const float v = g[j], z = w[s.perm[j]];
          d = fmaf(v, z, d);
          gg = fmaf(v, v, gg);
          mm = fmaf(z, z, mm);
          top = fmaxf(top, fabsf(v));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          d += __shfl_xor_sync(0xffffffffu, d, o);
          gg += __shfl_xor_sync(0xffffffffu, gg, o);
          mm += __shfl_xor_sync(0xffffffffu, mm, o);
          top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        }
        if (gg > 0.f && mm > 0.f) x += d * rsqrtf(gg) * rsqrtf(mm);
        if (side == 0) {
          int first = 4 * kCoreMaxDim;                       // 2 x column + (negative)
          for (int j = lane; j < r; j += 32)
            if (fabsf(g[j]) >= 0.9f * top) first = min(first, 2 * s.perm[j] + (g[j] < 0.f ? 1 : 0));
          first = __reduce_min_sync(0xffffffffu, first);
          turn = first & 1 ? -1.f : 1.f;
        }
      }
      if (lane == 0) out[c0 + i] = fabsf(x) > kSignFloor ? x : turn;
    }
  }
}

// Bond core, one cluster per bond.  Bound: the FP64 pipe (T_core = R1 R2^T, T Q
// and the FP64 Jacobi: 2 multiply-adds per clock and SM) and the shared-memory
// bandwidth of the FP32 Jacobi, both spread over the cluster's SMs; one CTA
// per bond left 150 of 152 SMs idle on a small grid and kept the Jacobi's
// columns in L2.  Core class of a saturated layer, one CTA -> cluster -> columns in
// registers (512 threads): 3x3 chi = 100 652 -> 93 -> 80 ms, 4x4 chi = 64 197 -> 39 ->
// 23 ms, 3x5 chi = 27 29.5 -> 13 -> 7.8 ms, 4x4 chi = 12 in FP64 30 -> 7.3 -> 3.9 ms.
__global__ void __launch_bounds__(kCoreThreads, 1)
k_core(const CoreItem* __restrict__ items, int* ival, int* flags_base, int csize) {
  const CoreItem it = items[blockIdx.x / csize];
  Cta ct;
  ct.rank = blockIdx.x % csize;
  ct.size = csize;
  ct.tid = (long long)ct.rank * blockDim.x + threadIdx.x;
  ct.nthr = (long long)csize * blockDim.x;
  int* flags = flags_base + it.inst;
  const int chic = ival[it.chi_idx];
  const int rg = ival[it.rg_idx];
  const int r = rg * chic;
  const int n = 4 * chic;
  const int k1 = ival[it.rank1_idx], k2 = ival[it.rank2_idx];
  const int rmax = it.rmax;
  double* R2t = it.work;                          // R2^T: r x k2, rows in R1's pivot order; later scratch
  double* Tc = it.work + (long long)rmax * rmax;  // column-major working matrix
  double* V = Tc + (long long)rmax * rmax;        // Jacobi right vectors
  double* Z = V + (long long)rmax * rmax;         // triangular-solve results
  int* cflag = reinterpret_cast<int*>(it.work + (long long)4 * rmax * rmax);   // 8 ints
  double* cnorm = it.work + (long long)4 * rmax * rmax + 4;                    // column norms (rmax)
  extern __shared__ __align__(16) unsigned char core_sh[];
  __shared__ double sv[2 * 4 * 128 + 8];
  __shared__ int order[4 * 128];
  __shared__ int sh_capped;
  const int lane = threadIdx.x & 31;
  const long long gw = ct.tid >> 5, ngw = ct.nthr >> 5;   // warps of the cluster
  if (threadIdx.x == 0) sh_capped = 0;
  if (ct.rank == 0 && threadIdx.x < 8) cflag[threadIdx.x] = 0;
  __shared__ float mold[2][128];                   // square roots of the old messages' diagonals
  for (int c = threadIdx.x; c < chic; c += blockDim.x) {
    mold[0][c] = sqrtf((float)fmax(it.msg12[(long long)c * it.chimax + c], 0.0));
    mold[1][c] = sqrtf((float)fmax(it.msg21[(long long)c * it.chimax + c], 0.0));
  }
  for (int q = threadIdx.x; q < r; q += blockDim.x) order[it.perm1[q]] = q;   // position in R1's pivot order
  __syncthreads();
  for (long long e = ct.tid; e < (long long)k2 * r; e += ct.nthr) {
    const int b = (int)(e / r), q = (int)(e % r);
    R2t[(long long)order[it.perm2[q]] * k2 + b] = (q >= b) ? it.T2[(long long)b * it.ldt2 + q] : 0.0;
  }
  cta_sync(ct);
  // Tcore = R1 R2^T (k1 x k2).  Work on the orientation with m >= n columns.
  const bool tr = k1 < k2;             // if so, decompose Tcore^T
  const int M = tr ? k2 : k1, N = tr ? k1 : k2;
  for (long long e = ct.tid; e < (long long)k1 * k2; e += ct.nthr) {
    const int a = (int)(e / k2), b = (int)(e % k2);
    double s = 0.0;
    const double* t1 = it.T1 + (long long)a * it.ldt1;
#pragma unroll 8
    for (int q = a; q < r; ++q) s = fma(t1[q], R2t[(long long)q * k2 + b], s);
    // column-major M x N storage of Tcore (or its transpose), and a copy (the
    // mixed path multiplies it by its FP64 subspace basis)
    const long long o = !tr ? (long long)b * M + a : (long long)a * M + b;
    Tc[o] = s;
    V[o] = s;
  }
  cta_sync(ct);
  // norms of the columns of a (len x cols, column-major) -> cnorm
  auto col_norms = [&](auto* a, int len, int cols) {
    for (long long j = gw; j < cols; j += ngw) {
      double s = 0.0;
      for (int i = lane; i < len; i += 32) { const double x = (double)a[j * len + i]; s = fma(x, x, s); }
      s = warp_sum(s);
      if (lane == 0) cnorm[j] = sqrt(s);
    }
    cta_sync(ct);
  };
  // descending order of sv[0 .. cols), NaN last, so that any input gives a
  // permutation (every order[] slot written once)
  auto rank_order = [&](int cols) {
    for (int j = threadIdx.x; j < cols; j += blockDim.x) {
      int rk = 0;
      const long long kj = mag_key(sv[j]);
      for (int i = 0; i < cols; ++i) {
        const long long ki = mag_key(sv[i]);
        if (ki > kj || (ki == kj && i < j)) ++rk;
      }
      order[rk] = j;
    }
    __syncthreads();
  };
  // columns the FP64 Jacobi below works on (all N, or the mixed path's subspace)
  int NK = N;
  __shared__ double sh_fro;
  if (it.mixed_svd) {
    // FP32 one-sided Jacobi with accumulated right vectors V32 (in the R2
    // block, free until the reconstruct step) finds the dominant right
    // singular subspace to FP32 accuracy.  Its leading NK = chimax + margin
    // directions are re-orthonormalised in FP64 (Cholesky QR; V32 itself is
    // orthogonal only to ~1e-5 after thousands of FP32 rotations) and the FP64
    // Jacobi then runs on T Q (M x NK) instead of T (M x N): the singular
    // values of T Q are those of T restricted to an exactly orthonormal basis,
    // so the kept values carry no error from V32's non-orthogonality, and the
    // FP64 work (GB300's FP64 rate is ~1/64 of its FP32 rate) drops by
    // (N / NK)^2 per sweep.  The columns are then nearly orthogonal, so few
    // FP64 sweeps follow.  Values past NK (never kept: NK > chimax) keep their
    // FP32 estimates for the diagnostic spectrum; the discarded weight of the
    // truncation uses ||T||_F^2 computed in FP64.
    float* T32 = reinterpret_cast<float*>(R2t);
    float* V32 = T32 + (long long)M * N;
    col_norms(Tc, M, N);
    double f2 = 0.0;
    for (int j = threadIdx.x; j < N; j += blockDim.x) f2 = fma(cnorm[j], cnorm[j], f2);
    {
      __shared__ double fr2[32];
      f2 = block_sum(f2, fr2);
    }
    if (threadIdx.x == 0) sh_fro = f2;
    __syncthreads();
    // the copy is scaled by a power of two to a norm in [1, 2): its squares stay
    // in FP32's range whatever the scale of the site tensors
    const int t_exp = sh_fro > 0.0 && isfinite(sh_fro) ? ilogb(sqrt(sh_fro)) : 0;
    for (long long e = ct.tid; e < (long long)M * N; e += ct.nthr) T32[e] = (float)scalbn(Tc[e], -t_exp);
    cta_sync(ct);
    __shared__ int sh_capped32;   // a capped FP32 pass only costs FP64 sweeps below
    const int sw32 = jacobi_cluster<float>(T32, M, N, V32, 60, &sh_capped32, 0.0, ct, cflag, cnorm, core_sh);
    if (ct.rank == 0 && threadIdx.x < 8) cflag[threadIdx.x] = 0;
    if (ct.rank == 0 && threadIdx.x == 0 && it.sweeps) it.sweeps[0] = sw32;
    // FP32 singular-value estimates (unsorted at sv[j]) and their order
    col_norms(T32, M, N);
    for (int j = threadIdx.x; j < N; j += blockDim.x) sv[j] = scalbn(cnorm[j], t_exp);
    __syncthreads();
    rank_order(N);
    for (int c = threadIdx.x; c < N; c += blockDim.x) sv[512 + c] = sv[order[c]];   // sorted FP32 values
    const int margin = it.chimax / 4 > 16 ? it.chimax / 4 : 16;
    NK = it.chimax + margin < N ? it.chimax + margin : N;
    // Q = leading NK columns of V32 in FP64 (N x NK, column-major, in Z)
    double* Qk = Z;
    for (long long e = ct.tid; e < (long long)N * NK; e += ct.nthr) {
      const int c = (int)(e / N), i = (int)(e - (long long)c * N);
      Qk[e] = (double)V32[(long long)order[c] * N + i];
    }
    cta_sync(ct);
    // Cholesky QR: G = Q^T Q = L L^T (lower triangle of G in the Tc block), Q <- Q L^-T
    double* G = Tc;
    for (long long pq = gw; pq < (long long)NK * NK; pq += ngw) {
      const int a = (int)(pq / NK), b = (int)(pq - (long long)a * NK);
      if (b > a) continue;
      const double* qa = Qk + (long long)a * N;
      const double* qb = Qk + (long long)b * N;
      double acc = 0.0;
      for (int i = lane; i < N; i += 32) acc = fma(qa[i], qb[i], acc);
      acc = warp_sum(acc);
      if (lane == 0) G[(long long)a * NK + b] = acc;
    }
    cta_sync(ct);
    // every CTA factors its own copy: the lower triangle packed in shared memory
    double* L = reinterpret_cast<double*>(core_sh);        // NK (NK + 1) / 2 <= 160 * 161 / 2 doubles
    for (int e = threadIdx.x; e < NK * NK; e += blockDim.x) {
      const int i = e / NK, l = e - i * NK;
      if (l <= i) L[i * (i + 1) / 2 + l] = G[e];
    }
    __syncthreads();
    double* Li = reinterpret_cast<double*>(core_sh) + 160 * 161 / 2;   // reciprocal diagonals
    for (int j = 0; j < NK; ++j) {
      const int jj = j * (j + 1) / 2;
      if (threadIdx.x == 0) {
        L[jj + j] = sqrt(L[jj + j]);
        Li[j] = 1.0 / L[jj + j];
      }
      __syncthreads();
      const double dinv = Li[j];
      for (int i = j + 1 + threadIdx.x; i < NK; i += blockDim.x) L[i * (i + 1) / 2 + j] *= dinv;
      __syncthreads();
      for (int i = j + 1 + (int)(threadIdx.x >> 5); i < NK; i += (int)(blockDim.x >> 5)) {
        const double lij = L[i * (i + 1) / 2 + j];
        for (int l = j + 1 + lane; l <= i; l += 32) L[i * (i + 1) / 2 + l] -= lij * L[l * (l + 1) / 2 + j];
      }
      __syncthreads();
    }
    for (long long i = ct.tid; i < N; i += ct.nthr) {   // row i of Q solves x L^T = q
      for (int c = 0; c < NK; ++c) {
        double x = Qk[(long long)c * N + i];
        const double* lc = L + c * (c + 1) / 2;
#pragma unroll 8
        for (int l = 0; l < c; ++l) x -= Qk[(long long)l * N + i] * lc[l];
        Qk[(long long)c * N + i] = x * Li[c];
      }
    }
    cta_sync(ct);
    // Tc <- T Q (M x NK, column-major), T = the copy in V
    for (long long e = ct.tid; e < (long long)M * NK; e += ct.nthr) {
      const int c = (int)(e / M), i = (int)(e - (long long)c * M);
      const double* qc = Qk + (long long)c * N;
      double acc = 0.0;
#pragma unroll 8
      for (int k = 0; k < N; ++k) acc = fma(V[(long long)k * M + i], qc[k], acc);
      Tc[e] = acc;
    }
    cta_sync(ct);
  }
  {   // FP64 one-sided Jacobi on Tcore (or on its restriction T Q)
    // mixed path: the rotations W64 (NK x NK) are accumulated in the V block
    // (the copy of T is no longer needed); the right vectors are then Q W64
    // the right vectors are always accumulated (V): recovering them as
    // T^T u / s would carry the columns' absolute rounding (~1e-16 of the
    // largest) divided by s^2, which for kept values near eps_cut (1e-11 of
    // the largest) leaves nothing of the vector
    const int sw64 = jacobi_cluster<double>(Tc, M, NK, V, 60, &sh_capped, 1e-17, ct, cflag, cnorm, core_sh);
    if (ct.rank == 0 && threadIdx.x == 0 && it.sweeps) {
      it.sweeps[1] = sw64;
      if (!it.mixed_svd) it.sweeps[0] = 0;
    }
    // singular values (column norms) and descending order
    col_norms(Tc, M, NK);
    for (int j = threadIdx.x; j < NK; j += blockDim.x) sv[j] = cnorm[j];
    __syncthreads();
    rank_order(NK);
  }
  const double s0 = NK > 0 ? sv[order[0]] : 0.0;
  // truncation, Eq. 11
  __shared__ int sh_chi;
  __shared__ double sh_sum, sh_nrm;
  if (threadIdx.x == 0) {
    int cnt = 0;
    double tot = 0.0;
    for (int i = 0; i < NK; ++i) {
      double s = sv[order[i]];
      tot += s * s;
      if (s >= it.eps_cut * s0 && s > 0.0) ++cnt;
    }
    if (it.mixed_svd) tot = sh_fro;
    int chi = cnt < it.chimax ? cnt : it.chimax;
    if (chi < 1) chi = 1;
    double kept = 0.0, ksum = 0.0;
    for (int i = 0; i < chi; ++i) { double s = sv[order[i]]; kept += s * s; ksum += s; }
    sh_chi = chi;
    sh_sum = ksum;
    sh_nrm = sqrt(kept);
    if (ct.rank == 0) {
      *it.disc = tot > 0.0 ? (tot - kept) / tot : 0.0;
      ival[it.new_idx] = chi;
      *it.nsv = N;
      if (!(s0 > 0.0) || !isfinite(s0)) atomicOr(flags, 2);
      // stored psi = true psi * exp(-sigma); the raw sqrt(S) split gives both
      // sites half of the pair's combined scale plus the normalisation of W
      const double ls = 0.5 * log(ksum) + 0.5 * (*it.sigma1 + *it.sigma2);
      *it.sigma1 = ls;
      *it.sigma2 = ls;
    }
    if (sh_capped) atomicOr(flags, 4);
  }
  __syncthreads();
  const int chi = sh_chi;
  // per kept value c: lambda_c, and the factor of its vector in W, sqrt(s_c) / sqrt(sum s),
  // divided by s_c for the side whose vectors are the unscaled columns
  __shared__ double lam[128], fac[2][128];
  for (int c = threadIdx.x; c < chi; c += blockDim.x) {
    const double sc = sv[order[c]];
    lam[c] = sc / sh_nrm;
    fac[0][c] = sqrt(sc / sh_sum);
    fac[1][c] = sc > 0.0 ? fac[0][c] / sc : 0.0;
  }
  __syncthreads();
  for (long long i = ct.tid; i < it.chimax; i += ct.nthr) it.lam[i] = (i < chi) ? lam[i] : 0.0;
  for (long long i = ct.tid; i < N; i += ct.nthr) it.svals[i] = i < NK ? sv[order[i]] : sv[512 + i];
  // messages diag(lambda)
  for (long long e = ct.tid; e < (long long)it.chimax * it.chimax; e += ct.nthr) {
    const int i = (int)(e / it.chimax), j = (int)(e % it.chimax);
    const double x = (i == j && i < chi) ? lam[i] : 0.0;
    it.msg12[e] = x;
    it.msg21[e] = x;
  }
  double* Vr = R2t;
  if (it.mixed_svd) {
    // Right (N-space) vectors of the kept pairs: v_c = Q W64 e_order[c] (N x chi,
    // column-major, in the R2 block).  These are the Ritz vectors of the
    // subspace, so T v_c = s_c u_c holds exactly for every kept pair; recovering
    // them as T^T u_c / s_c instead would divide the subspace's FP32-level
    // residual by s_c^2 for values near the FP32 resolution (~1e-7 of the largest).
    for (long long e = ct.tid; e < (long long)N * chi; e += ct.nthr) {
      const int c = (int)(e / N), a = (int)(e - (long long)c * N);
      const double* w = V + (long long)order[c] * NK;
      double acc = 0.0;
#pragma unroll 8
      for (int l = 0; l < NK; ++l) acc = fma(Z[(long long)l * N + a], w[l], acc);
      Vr[e] = acc;
    }
  }
  cta_sync(ct);
  // Signs of the singular pairs -> cnorm; msh[side][e]: what the side's old positive
  // vector brings to column e = (c, kappa) of X.
  {
    float* msh = reinterpret_cast<float*>(core_sh) + kSignSmem;
    for (int e = threadIdx.x; e < 2 * r; e += blockDim.x) {
      const int side = e >= r, col = e - side * r;
      msh[e] = mold[side][col / rg] * (float)(side == 0 ? it.FA : it.FB)[(col % rg) * 16];
    }
    // columns of Tc are s_c times their side's vectors
    auto vec = [&](int side, int c) -> const double* {
      if ((side == 0) != tr) return Tc + (long long)order[c] * M;
      return it.mixed_svd ? Vr + (long long)c * N : V + (long long)order[c] * N;
    };
    auto ex = [&](int side, int c) { return (side == 0) != tr ? (__double2hiint(sv[order[c]]) >> 20) & 0x7ff : 1023; };
    pair_signs({it.T1, it.perm1, it.ldt1, k1}, {it.T2, it.perm2, it.ldt2, k2}, r, chi, vec, ex, msh, ct, cnorm,
               reinterpret_cast<float*>(core_sh));
  }
  // For each side: Z_s = T_s11^{-1} (singular vectors of that side) sqrt(s) / sqrt(sum s);
  // side 1 vectors: left vectors of Tcore (rows of R1 space, length k1), side 2
  // vectors: right vectors (length k2).  Both sides at once, the columns
  // shared out over the CTAs, each solved in blocks of 32 rows: the rows of a
  // block one after another, then their contribution to all rows above as one
  // product (one dependent chain of 32 rows at a time instead of ks).
  // Z of side s: ks x chi column-major at Z + s rmax chimax (rmax = 4 chimax).
  double* Zs[2] = {Z, Z + (long long)rmax * it.chimax};
  {
    constexpr int kZld = kCoreMaxDim + 1;                  // odd: lanes on one row of several columns
    // reciprocal diagonals of both triangles
    double* di = reinterpret_cast<double*>(core_sh + kCoreSmem) - 2 * kCoreMaxDim;
    for (int a = threadIdx.x; a < k1; a += blockDim.x) di[a] = 1.0 / it.T1[(long long)a * it.ldt1 + a];
    for (int a = threadIdx.x; a < k2; a += blockDim.x) di[kCoreMaxDim + a] = 1.0 / it.T2[(long long)a * it.ldt2 + a];
    double* zc = reinterpret_cast<double*>(core_sh);       // this CTA's columns, ks each
    const int fit = ((int)(kCoreSmem / sizeof(double)) - 2 * kCoreMaxDim) / kZld;   // 45 columns at a time
    const int total = 2 * chi;
    const int per = min(fit, (total + ct.size - 1) / ct.size);
    for (int g0 = ct.rank * per; g0 < total; g0 += ct.size * per) {
      for (int side = 0; side < 2; ++side) {
        const int c0 = max(g0 - side * chi, 0), c1 = min(g0 + per - side * chi, chi);
        if (c0 >= c1) continue;
        const int nc = c1 - c0;
        const int ks = side == 0 ? k1 : k2;
        const double* Ts = side == 0 ? it.T1 : it.T2;
        const int ldts = side == 0 ? it.ldt1 : it.ldt2;
        // if (!tr): left vectors = columns of Tc / s (length M = k1), right = V (length N = k2)
        // if (tr):  left vectors = V (length N = k1), right = columns of Tc / s (length M = k2)
        const bool from_cols = (side == 0) != tr;
        __syncthreads();
        for (int e = threadIdx.x; e < ks * nc; e += blockDim.x) {
          const int c = e / ks, a = e - c * ks;
          const int j = order[c0 + c];
          double x;
          if (from_cols) x = Tc[(long long)j * M + a];
          else if (it.mixed_svd) x = Vr[(long long)(c0 + c) * N + a];   // Ritz right vector (above)
          else x = V[(long long)j * N + a];                             // accumulated right vector j
          zc[c * kZld + a] = x * fac[from_cols ? 1 : 0][c0 + c];
        }
        __syncthreads();
        for (int b1 = ks; b1 > 0; b1 -= 32) {
          const int b0 = b1 > 32 ? b1 - 32 : 0;
          // the block's own rows: one warp per column, lane = row
          for (int c = threadIdx.x >> 5; c < nc; c += (int)(blockDim.x >> 5)) {
            double* z = zc + c * kZld;
            double x = b0 + lane < b1 ? z[b0 + lane] : 0.0;
            for (int a = b1 - 1; a >= b0; --a) {
              const double y = __shfl_sync(0xffffffffu, x, a - b0) * di[side * kCoreMaxDim + a];
              if (b0 + lane == a) x = y;
              else if (b0 + lane < a) x -= Ts[(long long)(b0 + lane) * ldts + a] * y;
            }
            if (b0 + lane < b1) z[b0 + lane] = x;
          }
          __syncthreads();
          for (int e = threadIdx.x; e < b0 * nc; e += blockDim.x) {
            const int a = e / nc, c = e - a * nc;
            const double* trow = Ts + (long long)a * ldts;
            double* z = zc + c * kZld;
            double acc = z[a];
#pragma unroll 8
            for (int b = b0; b < b1; ++b) acc -= trow[b] * z[b];
            z[a] = acc;
          }
          __syncthreads();
        }
        for (int e = threadIdx.x; e < ks * nc; e += blockDim.x) {
          const int c = e / ks, a = e - c * ks;
          Zs[side][(long long)(c0 + c) * ks + a] = zc[c * kZld + a];
        }
      }
    }
  }
  cta_sync(ct);
  __shared__ float turn[128];
  for (int c = threadIdx.x; c < chi; c += blockDim.x) turn[c] = (float)cnorm[c];
  // Y[(c,kappa), c'] = Z[q, c'] at original column perm[q] (zero for q >= ks)
  // W[(c,p), (c',p')] = sum_kappa F_kappa[p', p] Y[(c,kappa), c']
  for (int side = 0; side < 2; ++side) {
    const int ks = side == 0 ? k1 : k2;
    const int* perms = side == 0 ? it.perm1 : it.perm2;
    const double* Fs = side == 0 ? it.FA : it.FB;
    double* W = side == 0 ? it.W1 : it.W2;
    __syncthreads();
    for (int q = threadIdx.x; q < r; q += blockDim.x) order[perms[q]] = q;   // position of each original column
    __syncthreads();
    const int np = 4 * chi;
    for (long long e = ct.tid; e < (long long)n * np; e += ct.nthr) {
      const int row = (int)(e / np), col = (int)(e % np);
      const int cc = row / 4, p = row % 4, c2 = col / 4, p2 = col % 4;
      double x = 0.0;
      for (int kk = 0; kk < rg; ++kk) {
        const int q = order[cc * rg + kk];
        const double y = q < ks ? Zs[side][(long long)c2 * ks + q] : 0.0;
        x += Fs[kk * 16 + p2 * 4 + p] * y;
      }
      W[(long long)row * it.ldw + col] = turn[c2] < 0.f ? -x : x;
    }
  }
}

// four blocks of rmax^2, the cluster's flags, column norms
size_t core_work_doubles(int rmax) { return (size_t)4 * rmax * rmax + 4 + rmax; }

// CTAs per core: as many (up to eight) as leave every bond its own SMs; long cores
// (chi_max > 32) may fill the chip three times over (the 50 bonds of a 10x10
// colour: eight each).  A batch of many small cores runs one or two CTAs each.
static int core_cluster(int n_items, int chimax) {
  const int most = chimax > 32 ? 3 * 152 : 152;
  for (int c = 8; c > 1; c /= 2)
    if (chimax > 8 && n_items * c <= most) return c;
  return 1;
}

cudaError_t launch_core(const CoreItem* items, int n_items, int chimax, int* ival, int* flags_base, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  const int csize = core_cluster(n_items, chimax);
  cudaError_t e = cudaFuncSetAttribute(k_core, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCoreSmem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_items * csize);
  cfg.blockDim = dim3(kCoreThreads);
  cfg.dynamicSmemBytes = kCoreSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = csize;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, k_core, items, ival, flags_base, csize);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace pepo

namespace pepo {
// ============================================================ message eigen
// The square roots of a message's eigenvalues scale the rotated legs (they
// are the weights of every Gram that sums over the leg) and divide the Gram
// of that leg back out, so they are floored at kSqrtEigFloor of the largest:
// an eigenvalue below 1e-12 of the largest counts as 1e-12 of it, which
// moves no message by more than that relative amount.
constexpr double kSqrtEigFloor = 1e-6;
__device__ void floor_sqrt_eigs(double* sd, int n, double* red) {
  __syncthreads();
  double m = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) m = fmax(m, sd[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) m = fmax(m, red[i]);
  const double lo = kSqrtEigFloor * (m > 0.0 ? m : 1.0);
  for (int j = threadIdx.x; j < n; j += blockDim.x) sd[j] = fmax(sd[j], lo);
  __syncthreads();
}

// Vs = diag(sd) Vt: the BP rotation of a leg scaled by the square roots of
// the message's eigenvalues
__device__ void scaled_rotation(const EnvEigItem& it, int n) {
  if (!it.Vs) return;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, j = e - i * n;
    it.Vs[i * it.ld + j] = it.sqrtD[i] * it.Vt[i * it.ld + j];
  }
}

// M (symmetrised, PSD) -> one-sided Jacobi on its columns: M V = U S with
// S = |eigenvalues| and V the eigenvectors (U = V up to signs of numerically
// zero eigenvalues).  Outputs Vt (row i = column i of V) and sqrt(S).  FP32
// (R = float, FP32-storage modes): the eigenbasis only rotates FP32 tensors.
// The matrices live in shared memory; FP64 ones that do not fit (chi > 112) in
// the item's workspace.
constexpr size_t kEigSmem = (size_t)220 * 1024;
template <typename R>
__host__ __device__ inline size_t eig_smem(int chimax) {   // norms, A and V
  return sizeof(R) == 4 ? sizeof(float) * (128 + 2 * (size_t)chimax * jac_ld(chimax))
                        : sizeof(double) * (128 + 2 * (size_t)chimax * chimax);
}
template <typename R>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 1024 : 512)
k_env_eig(const EnvEigItem* __restrict__ items, const int* ival, int chimax) {
  const EnvEigItem it = items[blockIdx.x];
  const int n = ival[it.chi_idx];
  extern __shared__ __align__(16) unsigned char eig_sh[];
  __shared__ double red[32], sq[128];
  __shared__ int capped;
  if (threadIdx.x == 0) capped = 0;
  R* nrm = reinterpret_cast<R*>(eig_sh);                   // 128 values
  R* A = eig_smem<R>(chimax) <= kEigSmem ? nrm + 128 : reinterpret_cast<R*>(it.work);
  int ld;
  R* V;
  if constexpr (sizeof(R) == 4) { ld = jac_ld(n); V = A + n * ld; }
  else { ld = 2 * n; V = A + n; }
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, j = e - i * n;
    A[j * ld + i] = (R)(0.5 * (it.M[i * it.ld + j] + it.M[j * it.ld + i]));
  }
  __syncthreads();
  if constexpr (sizeof(R) == 4) {
    if (n <= 32) jacobi_block_l<float, 8, 4>(A, n, ld, V, nrm, 60, &capped);
    else if (n <= 64) jacobi_block_l<float, 16, 4>(A, n, ld, V, nrm, 60, &capped);
    else jacobi_block_l<float, 16, 8>(A, n, ld, V, nrm, 60, &capped);
  } else {
    __shared__ JacRound jr;
    if (n <= 8) jacobi_block_l<double, 8, 1>(A, n, ld, V, nrm, 60, &capped);
    else if (n <= 16) jacobi_block_l<double, 16, 1>(A, n, ld, V, nrm, 60, &capped);
    else jacobi_block64(A, n, nrm, 60, &capped, jr);
  }
  for (int j = threadIdx.x >> 5; j < n; j += (int)(blockDim.x >> 5)) {
    double s = 0.0;
    for (int i = threadIdx.x & 31; i < n; i += 32) s = fma((double)A[j * ld + i], (double)A[j * ld + i], s);
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) sq[j] = s;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < n; j += blockDim.x) it.sqrtD[j] = sqrt(sqrt(sq[j]));   // of |lambda_j| = ||A v_j||
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, j = e - i * n;
    it.Vt[i * it.ld + j] = (double)V[i * ld + j];          // row i of Vt = column i of V
  }
  floor_sqrt_eigs(it.sqrtD, n, red);
  scaled_rotation(it, n);
}

template <typename R>
static cudaError_t launch_eig(const EnvEigItem* items, int n_items, int chimax, const int* ival, cudaStream_t s) {
  const size_t want = eig_smem<R>(chimax);
  const size_t smem = want <= kEigSmem ? want : sizeof(R) * 128;
  cudaError_t e = cudaFuncSetAttribute(k_env_eig<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // FP32: every pair of a round its lanes; FP64: a warp per pair of columns
  const int pairs = (chimax + 1) / 2;
  const int threads = sizeof(R) == 4 ? std::max(64, (jac_lanes(chimax) * pairs + 31) / 32 * 32)
                                     : std::min(512, std::max(128, 32 * pairs));
  k_env_eig<R><<<n_items, threads, smem, s>>>(items, ival, chimax);
  return cudaGetLastError();
}

cudaError_t launch_env_eig(const EnvEigItem* items, int n_items, int chimax, int fp32, const int* ival,
                           cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  return fp32 ? launch_eig<float>(items, n_items, chimax, ival, s) : launch_eig<double>(items, n_items, chimax, ival, s);
}

// out = V G' V^T = Vt^T (G' Vt), G' = G / (sd sd^T).  A block forms a strip of the
// output's columns: its strip of G' Vt in shared memory, then Vt^T times that, so
// the strips of a message need nothing from each other.  Bound: the FP64 pipe
// (4 n^3 operations a message), shared by as many SMs as the strips fill; the
// divisions by sd are n per block (they were one per product, ~16
// multiply-adds each, on one SM per message: 2.7 ms a launch at chi = 100, now
// 0.2).
__global__ void __launch_bounds__(256)
k_rotate_back(const RotItem* __restrict__ items, const int* ival) {
  const RotItem it = items[blockIdx.x];
  const int n = ival[it.chi_idx];
  const int w = (n + gridDim.y - 1) / gridDim.y;
  const int j0 = blockIdx.y * w, nj = min(w, n - j0);
  if (nj <= 0) return;
  extern __shared__ __align__(16) double sm[];
  double* T = sm;            // n x nj: T = G' Vt[:, j0 ..]
  double* B = sm + n * w;    // n x nj: Vt[:, j0 ..] with row k divided by sd[k]
  double* isd = B + n * w;   // 1 / sd
  for (int i = threadIdx.x; i < n; i += blockDim.x) isd[i] = it.sd ? 1.0 / it.sd[i] : 1.0;
  __syncthreads();
  for (int e = threadIdx.x; e < n * nj; e += blockDim.x) {
    const int k = e / nj, j = e - k * nj;
    B[e] = it.Vt[k * it.ld + j0 + j] * isd[k];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n * nj; e += blockDim.x) {
    const int i = e / nj, j = e - i * nj;
    const double* g = it.G + i * it.ld;
    double s = 0.0;
#pragma unroll 4
    for (int k = 0; k < n; ++k) s = fma(g[k], B[k * nj + j], s);
    T[e] = s * isd[i];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n * nj; e += blockDim.x) {
    const int i = e / nj, j = e - i * nj;
    const double* v = it.Vt + i;
    double s = 0.0;
#pragma unroll 4
    for (int k = 0; k < n; ++k) s = fma(v[k * it.ld], T[k * nj + j], s);
    it.out[i * it.ld + j0 + j] = s;
  }
}

cudaError_t launch_rotate_back(const RotItem* items, int n_items, int chimax, const int* ival,
                               cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  // strips: enough blocks for two per SM, columns of a strip at least four
  int strips = ceil_div(2 * 152, n_items);
  strips = std::max(1, std::min(strips, std::min(16, chimax / 4)));
  if (strips < 2 && chimax > 96) strips = 2;   // two strips of chi^2 / strips doubles in shared memory
  const size_t smem = sizeof(double) * ((size_t)2 * chimax * ceil_div(chimax, strips) + chimax);
  cudaError_t e = cudaFuncSetAttribute(k_rotate_back, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  k_rotate_back<<<dim3(n_items, strips), 256, smem, s>>>(items, ival);
  return cudaGetLastError();
}
}  // namespace pepo
