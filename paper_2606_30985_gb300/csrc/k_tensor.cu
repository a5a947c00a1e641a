// HBM-bound tensor kernels of the bond update and of BP.
//
//   k_gram_rows32/64 cv^T cv (Eq. 10, Cholesky-QR Gram)
//   k_gram_exact     cv^T cv of FP32 data to FP64 accuracy (FP32 storage: the sites of the
//                    Householder side of Eq. 10 and those whose Gram fails its test)
//   k_reconstruct, k_reconstruct32   psi_new = psi W written in the next update's layout
//                    (Sec. 2.5 steps 6-7 in Q-less form, Alg. 1 lines 9-12)
//   k_vec_pair, k_vec_contract   vector contractions of single-layer BP (Sec. 2.6)
//
// All sizes are read on the device (see common.cuh).  Accumulation: FP32
// storage accumulates with FP32 FMAs over short runs that go into two-float or
// FP64 sums, so long sums (up to chi^3 terms) keep far below the FP32 error
// (Sec. 4.2 "Gram matrix accumulation error": the paper's FP32 Gram loses
// m * eps; this does not).
#include "kernels.h"

namespace pepo {

__device__ inline void load_dims(const TView& v, const int* ival, int* d) {
#pragma unroll
  for (int k = 0; k < PEPO_MAXLEG; ++k) d[k] = (k < v.nlegs) ? ival[v.dim[k]] : 1;
}

// ======================================================================= copy
template <typename T>
__global__ void k_copy(const TView* __restrict__ items, const int* __restrict__ out_refs,
                       void* const* ptrs, const int* __restrict__ ival) {
  const TView v = items[blockIdx.y];
  int d[PEPO_MAXLEG];
  load_dims(v, ival, d);
  long long n = 4;
  for (int k = 0; k < v.nlegs; ++k) n *= d[k];
  const T* in = static_cast<const T*>(ptrs[v.ref]);
  T* out = static_cast<T*>(ptrs[out_refs[blockIdx.y]]);
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = in[i];
}

template <typename T>
cudaError_t launch_copy(const TView* items, const int* out_refs, int n_items, int grid_x,
                        void* const* ptrs, const int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  k_copy<T><<<dim3(grid_x, n_items), 256, 0, s>>>(items, out_refs, ptrs, ival);
  return cudaGetLastError();
}

// ================================================================ Gram (rows)
// Tiles of 64 x 64, the rows K split over blocks (gram_rows_splits).
constexpr int GR_T = 64;
constexpr int GR_BK = 16;
constexpr int GR_FLUSH = 256;   // FP32 run length before the two-float sum takes it

__device__ inline void tile_of(int t, int nt, int sym, int& ti, int& tj) {
  if (!sym) { ti = t / nt; tj = t - ti * nt; return; }
  // upper-triangular enumeration: row ti holds nt - ti tiles
  int r = 0, base = 0;
  while (r < nt && t >= base + (nt - r)) { base += nt - r; ++r; }
  ti = r; tj = r + (t - base);
}

// FP64 storage: bound by the FP64 pipe whatever the tile.
__global__ void __launch_bounds__(256)
k_gram_rows64(const GramRowsItem* __restrict__ items, int splits_max, int sym, void* const* ptrs,
              const int* __restrict__ ival) {
  const GramRowsItem it = items[blockIdx.z];
  if (it.active >= 0 && ival[it.active] == 0) return;
  int d[PEPO_MAXLEG];
  load_dims(it.x, ival, d);
  const int nl = it.x.nlegs;
  const int F = 4 * (nl > 0 ? d[nl - 1] : 1);
  long long K = 1;
  for (int i = 0; i + 1 < nl; ++i) K *= d[i];
  const int S = gram_rows_splits(K, splits_max);
  const int s = blockIdx.x % splits_max;
  const int t = blockIdx.x / splits_max;
  const int nt = ceil_div(F, GR_T);
  const int ntiles = sym ? nt * (nt + 1) / 2 : nt * nt;
  if (s >= S || t >= ntiles) return;
  int ti, tj;
  tile_of(t, nt, sym, ti, tj);
  const long long k0 = K * s / S, k1 = K * (s + 1) / S;
  const double* __restrict__ X = static_cast<const double*>(ptrs[it.x.ref]);
  __shared__ __align__(16) double Xs[GR_BK][GR_T];
  __shared__ __align__(16) double Ys[GR_BK][GR_T];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  for (long long kb = k0; kb < k1; kb += GR_BK) {
    for (int e = threadIdx.x; e < GR_BK * GR_T; e += blockDim.x) {
      int kk = e / GR_T, c = e - kk * GR_T;
      long long k = kb + kk;
      int fi = ti * GR_T + c, fj = tj * GR_T + c;
      bool okk = k < k1;
      Xs[kk][c] = (okk && fi < F) ? X[k * F + fi] : 0.0;
      Ys[kk][c] = (okk && fj < F) ? X[k * F + fj] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GR_BK; ++kk) {
      double xa[4], yb[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) xa[a] = Xs[kk][ty * 4 + a];
#pragma unroll
      for (int b = 0; b < 4; ++b) yb[b] = Ys[kk][tx * 4 + b];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = fma(xa[a], yb[b], acc[a][b]);
    }
    __syncthreads();
  }
  double* P = it.partial + (long long)s * F * F;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    int fi = ti * GR_T + ty * 4 + a;
    if (fi >= F) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int fj = tj * GR_T + tx * 4 + b;
      if (fj < F) P[(long long)fi * F + fj] = acc[a][b];
    }
  }
}

// 16-byte asynchronous copy of a quad, zeros where it lies outside
__device__ inline void copy_quad(void* dst, const void* src, bool live) {
  const int n = live ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(n)
               : "memory");
}

// FP32 storage.  64 x 64 tiles of the upper triangle; a chunk of 64 rows is
// copied asynchronously, three stages deep.  Two groups of 128 threads take 32
// rows of a chunk each, a thread 8 x 4 entries (32 multiply-adds per three
// 16-byte shared loads, two of them broadcasts), so the FP32 pipe bounds it;
// 4 x 4 entries and scalar, unpipelined loads ran at 18 TFLOP/s (class of a 4x4
// chi = 64 layer 17 -> 8.3 ms, 3x3 chi = 100 55 -> 25 ms).  Runs of 256
// terms in FP32 go into a two-float sum (within 1e-16 of the columns' norms of an FP64
// sum of the same runs, for 2^11 to 2^20 rows), the groups and splits into FP64.
constexpr int GF_K = 64;
constexpr int GF_STAGES = 3;

__global__ void __launch_bounds__(256, 2)
k_gram_rows32(const GramRowsItem* __restrict__ items, int splits_max, int sym, void* const* ptrs,
              const int* __restrict__ ival) {
  const GramRowsItem it = items[blockIdx.z];
  if (it.active >= 0 && ival[it.active] == 0) return;
  int d[PEPO_MAXLEG];
  load_dims(it.x, ival, d);
  const int nl = it.x.nlegs;
  const int F = 4 * (nl > 0 ? d[nl - 1] : 1);
  long long K = 1;
  for (int i = 0; i + 1 < nl; ++i) K *= d[i];
  const int S = gram_rows_splits(K, splits_max);
  const int sp = blockIdx.x % splits_max;
  const int nt = ceil_div(F, GR_T);
  if (sp >= S || (int)(blockIdx.x / splits_max) >= (sym ? nt * (nt + 1) / 2 : nt * nt)) return;
  int ti, tj;
  tile_of(blockIdx.x / splits_max, nt, sym, ti, tj);
  const bool diag = ti == tj;
  const long long k0 = K * sp / S, k1 = K * (sp + 1) / S;
  const float* __restrict__ X = static_cast<const float*>(ptrs[it.x.ref]);
  extern __shared__ __align__(16) float gf_sh[];       // stages of [X | Y], 64 rows x 64 columns each
  const int tid = threadIdx.x, g = tid >> 7, tx = tid & 15, ty = (tid >> 4) & 7;
  auto load = [&](int st, long long kb) {
    if (kb < k1) {
      float* xs = gf_sh + st * (2 * GF_K * GR_T);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = tid + 256 * u;                   // 64 rows x 16 quads
        const int row = e >> 4, q = 4 * (e & 15);
        const long long k = kb + row;
        const int ci = ti * GR_T + q, cj = tj * GR_T + q;
        const bool in = k < k1;
        copy_quad(xs + row * GR_T + q, in && ci < F ? X + k * F + ci : X, in && ci < F);
        if (!diag) copy_quad(xs + (GF_K + row) * GR_T + q, in && cj < F ? X + k * F + cj : X, in && cj < F);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[8][4];
  TwoFloat sum[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
  auto flush = [&]() {
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) { sum[a][b].take(acc[a][b]); acc[a][b] = 0.f; }
  };
#pragma unroll
  for (int st = 0; st < GF_STAGES - 1; ++st) load(st, k0 + st * GF_K);
  int st = 0, run = 0;
  for (long long kb = k0; kb < k1; kb += GF_K) {
    asm volatile("cp.async.wait_group %0;" ::"n"(GF_STAGES - 2) : "memory");
    __syncthreads();                                   // this chunk is in, the one before is consumed
    load(st == 0 ? GF_STAGES - 1 : st - 1, kb + (GF_STAGES - 1) * GF_K);
    const float* xs = gf_sh + st * (2 * GF_K * GR_T) + g * (GF_K / 2) * GR_T;
    const float* ys = diag ? xs : xs + GF_K * GR_T;
#pragma unroll 8
    for (int kk = 0; kk < GF_K / 2; ++kk) {
      float a8[8], b4[4];
      *reinterpret_cast<float4*>(a8) = *reinterpret_cast<const float4*>(xs + kk * GR_T + 4 * ty);
      *reinterpret_cast<float4*>(a8 + 4) = *reinterpret_cast<const float4*>(xs + kk * GR_T + 32 + 4 * ty);
      *reinterpret_cast<float4*>(b4) = *reinterpret_cast<const float4*>(ys + kk * GR_T + 4 * tx);
#pragma unroll
      for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(a8[a], b4[b], acc[a][b]);
    }
    run += GF_K / 2;
    if (run >= GR_FLUSH) { flush(); run = 0; }
    if (++st == GF_STAGES) st = 0;
  }
  flush();
  // the two groups' sums, then the split's tile
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  double* red = reinterpret_cast<double*>(gf_sh);
  if (g == 1)
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b)
        red[(4 * ty + (a & 3) + 32 * (a >> 2)) * GR_T + 4 * tx + b] = sum[a][b].value();
  __syncthreads();
  if (g == 0) {
    double* P = it.partial + (long long)sp * F * F;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const int r = 4 * ty + (a & 3) + 32 * (a >> 2), fi = ti * GR_T + r;
      if (fi >= F) continue;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int fj = tj * GR_T + 4 * tx + b;
        if (fj < F) P[(long long)fi * F + fj] = red[r * GR_T + 4 * tx + b] + sum[a][b].value();
      }
    }
  }
}

__global__ void k_gram_rows_reduce(const GramRowsItem* __restrict__ items, int splits_max, int sym,
                                   const int* __restrict__ ival) {
  const GramRowsItem it = items[blockIdx.y];
  if (it.active >= 0 && ival[it.active] == 0) return;
  int d[PEPO_MAXLEG];
  load_dims(it.x, ival, d);
  const int nl = it.x.nlegs;
  const int F = 4 * (nl > 0 ? d[nl - 1] : 1);
  long long K = 1;
  for (int i = 0; i + 1 < nl; ++i) K *= d[i];
  const int S = gram_rows_splits(K, splits_max);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < F * F; e += gridDim.x * blockDim.x) {
    int fi = e / F, fj = e - fi * F;
    int a = fi, b = fj;
    if (sym && (fi / GR_T) > (fj / GR_T)) { a = fj; b = fi; }
    double sum = 0.0;
    for (int s = 0; s < S; ++s) sum += it.partial[(long long)s * F * F + (long long)a * F + b];
    it.out[(long long)fi * it.ldo + fj] = sum;
  }
}

template <typename T>
cudaError_t launch_gram_rows(const GramRowsItem* items, int n_items, int tiles_max, int splits_max,
                             int sym, void* const* ptrs, const int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  dim3 grid(tiles_max * splits_max, 1, n_items);
  if constexpr (sizeof(T) == 8) {
    k_gram_rows64<<<grid, 256, 0, s>>>(items, splits_max, sym, ptrs, ival);
  } else {
    const size_t smem = sizeof(float) * GF_STAGES * 2 * GF_K * GR_T;
    cudaError_t e = cudaFuncSetAttribute(k_gram_rows32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_gram_rows32<<<grid, 256, smem, s>>>(items, splits_max, sym, ptrs, ival);
  }
  return cudaGetLastError();
}

cudaError_t launch_gram_rows_reduce(const GramRowsItem* items, int n_items, int fmax,
                                    int splits_max, int sym, const int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  int gx = ceil_div(fmax * fmax, 256);
  if (gx > 256) gx = 256;
  k_gram_rows_reduce<<<dim3(gx, n_items), 256, 0, s>>>(items, splits_max, sym, ival);
  return cudaGetLastError();
}


// ======================================================= exact Gram (rows)
// C = cv^T cv of FP32 data to the accuracy of FP64 sums, for the sites the branch
// rule of Eq. 10 sends to Householder and for those whose FP32-run Gram failed the
// trust test.  A pivoted Cholesky of this C finds every direction that keeps more
// than 1e-7 of the largest (1e-14 of the squares; the Gram's entries are within ~5e-16
// of the paired columns' norms at 64 rows and less above).
//
// Sum: the product's rounded part p and its rest q = ab - p; p goes into an
// accumulator s that starts at the anchor 3 P_i P_j, P the next power of two above the
// run's column norm, so by Cauchy-Schwarz s stays in one binade and what it leaves
// over, r, is at most 2^-23 P_i P_j.  The r go the same way into a second
// accumulator c, anchored 2^-17 lower, and what that leaves over (2^-40) and q into
// a third, d, in plain FP32: ten FP32 operations a term instead of one FP64
// multiply-add, which takes 64 issue slots here.  (With the r summed in plain FP32,
// four operations a term, an entry was 1e-12 off at 64 rows and a Cholesky took
// its noise for directions; class of a 4x4 chi = 64 layer 8.2 -> 17.3 ms, 3x3 chi = 100
// 20.9 -> 38.)  A run's 64 rows go into (S, U, W), each the rounding of the one
// before, the splits into FP64.  Columns are scaled to a largest magnitude in
// [1/2, 1) first (k_col_scale), so tiny tensors do not underflow.
//
// 64 x 64 tiles, 4 x 4 entries a thread (160 FP32 operations per two 16-byte
// shared loads: ALU-bound), 16-byte asynchronous copies one run ahead; U and W lie
// in shared memory, which leaves two blocks an SM.
// K splits: ~128 rows, two runs, each, at most kExactSplits, so that small sites fill the
// chip (a run takes a block 10 us; class of a 4x4 chi = 16 layer 0.92 ms with 512 rows,
// 0.44 with 128).
constexpr int GX_T = 64;
constexpr int GX_RUN = 64;
constexpr int kExactSplits = 60;
__device__ inline int exact_splits(long long K) { return (int)max(1ll, min(K / 128, (long long)kExactSplits)); }
constexpr float kGxLower = 1.f / 131072.f;   // 64 remainders of 2^-23 P_i P_j stay below 2^-17

__device__ inline float pow2f(int e) { return __int_as_float((min(max(e, -126), 127) + 127) << 23); }

// largest magnitude per column -> colmax (float bits, zeroed by the caller)
__global__ void __launch_bounds__(256)
k_col_scale(const GramRowsItem* __restrict__ items, int pass, int step, void* const* ptrs, const int* __restrict__ ival) {
  const GramRowsItem it = items[blockIdx.y];
  if (ival[it.active] != pass) return;
  int d[PEPO_MAXLEG];
  load_dims(it.x, ival, d);
  const int nl = it.x.nlegs;
  const int quads = nl > 0 ? d[nl - 1] : 1;            // F / 4
  const int F = 4 * quads;
  unsigned* cm = it.colmax;
  if (step == 0) {
    for (int c = threadIdx.x; c < F; c += blockDim.x) cm[c] = 0u;
    return;
  }
  long long K = 1;
  for (int i = 0; i + 1 < nl; ++i) K *= d[i];
  __shared__ unsigned sm[4 * 128];
  for (int c = threadIdx.x; c < F; c += blockDim.x) sm[c] = 0u;
  __syncthreads();
  const int rpb = 256 / quads;
  const int rr = threadIdx.x / quads, qd = threadIdx.x - rr * quads;
  if (rr < rpb) {
    const float* X = static_cast<const float*>(ptrs[it.x.ref]);
    unsigned m[4] = {0u, 0u, 0u, 0u};
    for (long long r = (long long)blockIdx.x * rpb + rr; r < K; r += (long long)gridDim.x * rpb) {
      const float4 v = *reinterpret_cast<const float4*>(X + r * F + 4 * qd);
      m[0] = max(m[0], __float_as_uint(fabsf(v.x)));
      m[1] = max(m[1], __float_as_uint(fabsf(v.y)));
      m[2] = max(m[2], __float_as_uint(fabsf(v.z)));
      m[3] = max(m[3], __float_as_uint(fabsf(v.w)));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (m[i]) atomicMax(&sm[4 * qd + i], m[i]);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < F; c += blockDim.x)
    if (sm[c]) atomicMax(&cm[c], sm[c]);
}

// exponent e with the column's largest magnitude in [2^(e-1), 2^e)
__device__ inline int col_exp(unsigned bits) { return (int)(bits >> 23) - 126; }

__global__ void __launch_bounds__(256, 2)
k_gram_exact(const GramRowsItem* __restrict__ items, int pass, void* const* ptrs, const int* __restrict__ ival) {
  const GramRowsItem it = items[blockIdx.z];
  if (ival[it.active] != pass) return;
  int d[PEPO_MAXLEG];
  load_dims(it.x, ival, d);
  const int nl = it.x.nlegs;
  const int F = 4 * (nl > 0 ? d[nl - 1] : 1);
  long long K = 1;
  for (int i = 0; i + 1 < nl; ++i) K *= d[i];
  const int S = exact_splits(K);
  const int sp = blockIdx.x % kExactSplits;
  const int nt = ceil_div(F, GX_T);
  if (sp >= S || (int)(blockIdx.x / kExactSplits) >= nt * (nt + 1) / 2) return;
  int ti, tj;
  tile_of(blockIdx.x / kExactSplits, nt, 1, ti, tj);
  const bool diag = ti == tj;
  const long long k0 = K * sp / S, k1 = K * (sp + 1) / S;
  const float* __restrict__ X = static_cast<const float*>(ptrs[it.x.ref]);
  // 2 buffers of [X tile | Y tile], 64 rows x 64 columns each; then U and W, 16 values a thread
  extern __shared__ __align__(16) float gx_sh[];
  __shared__ float nrm[2][2 * GX_T];                   // half sums of squares per column
  __shared__ float pw[2 * GX_T];                       // P per column
  __shared__ float sc[2 * GX_T];                       // column pre-scale 2^-e
  // A warp takes 32 x 16 entries, 8 x 4 threads; it has none outside the matrix or below
  // the diagonal.  Which of the four column strips it takes turns with the block, so that
  // the warps without entries are not all on one scheduler.
  const int tid = threadIdx.x, wr = tid >> 7, wc = ((tid >> 5) + 2 * wr + blockIdx.x) & 3;
  const int ty = 8 * wr + ((tid & 31) >> 2), tx = 4 * wc + (tid & 3);
  const bool live = ti * GX_T + 32 * wr < F && tj * GX_T + 16 * wc < F && (!diag || 32 * wr < 16 * wc + 16);
  if (tid < 2 * GX_T) {
    const int c = (tid < GX_T ? ti : tj) * GX_T + (tid & (GX_T - 1));
    sc[tid] = c < F ? pow2f(-col_exp(it.colmax[c])) : 0.f;
  }
  auto load = [&](int buf, long long kb) {
    float* xs = gx_sh + buf * (2 * GX_RUN * GX_T);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + 256 * u;                     // 64 rows x 16 quads
      const int row = e >> 4, qd = e & 15;
      const long long k = kb + row;
      const int ci = ti * GX_T + 4 * qd, cj = tj * GX_T + 4 * qd;
      const bool okk = k < k1;
      copy_quad(xs + row * GX_T + 4 * qd, okk && ci < F ? X + k * F + ci : X, okk && ci < F);
      if (!diag) copy_quad(xs + (GX_RUN + row) * GX_T + 4 * qd, okk && cj < F ? X + k * F + cj : X, okk && cj < F);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float S0[4][4];
  float* UW = gx_sh + 4 * GX_RUN * GX_T + tid;         // U at 512 e, W at 512 e + 256
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      S0[a][b] = 0.f;
      UW[512 * (4 * a + b)] = UW[512 * (4 * a + b) + 256] = 0.f;
    }
  if (k0 < k1) load(0, k0);
  int buf = 0;
  for (long long kb = k0; kb < k1; kb += GX_RUN, buf ^= 1) {
    if (kb + GX_RUN < k1) {
      load(buf ^ 1, kb + GX_RUN);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    float* xs = gx_sh + buf * (2 * GX_RUN * GX_T);
    float* ys = diag ? xs : xs + GX_RUN * GX_T;
    {   // scale the columns in place and sum their squares, half a column a thread
      const int c = tid & (GX_T - 1), half = (tid >> 6) & 1, isy = tid >> 7;
      if (!(isy && diag)) {
        float* col = (isy ? ys : xs) + c + half * (GX_RUN / 2) * GX_T;
        const float f = sc[isy * GX_T + c];
        float q = 0.f;
#pragma unroll 8
        for (int i = 0; i < GX_RUN / 2; ++i) {
          const float x = col[i * GX_T] * f;
          col[i * GX_T] = x;
          q = fmaf(x, x, q);
        }
        nrm[half][isy * GX_T + c] = q;
      }
    }
    __syncthreads();
    if (tid < 2 * GX_T) {
      const int c = diag ? (tid & (GX_T - 1)) : tid;
      const float q = (nrm[0][c] + nrm[1][c]) * 1.01f;
      const int e = (int)(__float_as_uint(q) >> 23) - 127;     // q < 2^(e + 1)
      pw[tid] = pow2f(max((e + 2) >> 1, -50));                 // P^2 > q
    }
    __syncthreads();
    if (live) {
      float s[4][4], c[4][4], d[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          s[a][b] = 3.f * (pw[ty * 4 + a] * pw[GX_T + tx * 4 + b]);
          c[a][b] = kGxLower * s[a][b];
          d[a][b] = 0.f;
        }
#pragma unroll 4
      for (int kk = 0; kk < GX_RUN; ++kk) {
        const float4 xa = *reinterpret_cast<const float4*>(xs + kk * GX_T + ty * 4);
        const float4 yb = *reinterpret_cast<const float4*>(ys + kk * GX_T + tx * 4);
        const float a4[4] = {xa.x, xa.y, xa.z, xa.w}, b4[4] = {yb.x, yb.y, yb.z, yb.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float p = __fmul_rn(a4[a], b4[b]);
            const float q = fmaf(a4[a], b4[b], -p);
            const float t = __fadd_rn(s[a][b], p);
            const float r = __fsub_rn(p, __fsub_rn(t, s[a][b]));
            const float u = __fadd_rn(c[a][b], r);
            d[a][b] += __fsub_rn(r, __fsub_rn(u, c[a][b]));
            d[a][b] += q;
            s[a][b] = t;
            c[a][b] = u;
          }
      }
      // the run's sum into (S, U, W)
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const float anchor = 3.f * (pw[ty * 4 + a] * pw[GX_T + tx * 4 + b]);
          float* uw = UW + 512 * (4 * a + b);
          TwoFloat hi, mid;                                      // c: what the sum leaves over
          hi.s = S0[a][b];
          hi.take(s[a][b] - anchor);                             // exact difference
          mid.s = uw[0];
          mid.take(c[a][b] - kGxLower * anchor);                 // exact too
          mid.take(hi.c);
          S0[a][b] = hi.s;
          uw[0] = mid.s;
          uw[256] += mid.c + d[a][b];
        }
    }
    __syncthreads();                                           // the buffer is refilled next
  }
  if (!live) return;
  double* Pt = it.partial + (long long)sp * F * F;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int fi = ti * GX_T + ty * 4 + a;
    if (fi >= F) continue;
    const int ei = col_exp(it.colmax[fi]);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int fj = tj * GX_T + tx * 4 + b;
      if (fj < F) {
        const float* uw = UW + 512 * (4 * a + b);
        const double v = (double)S0[a][b] + ((double)uw[0] + (double)uw[256]);
        Pt[(long long)fi * F + fj] = scalbn(v, ei + col_exp(it.colmax[fj]));
      }
    }
  }
}

// Sum of the splits, mirrored into the lower triangle; acct (2 doubles, may be
// null) accumulates the FLOPs (one multiply-add per entry of the triangle and
// row) and bytes (one read of the matrix), which only the device knows.
__global__ void k_gram_exact_reduce(const GramRowsItem* __restrict__ items, int pass, const int* __restrict__ ival,
                                    double* acct) {
  const GramRowsItem it = items[blockIdx.y];
  if (ival[it.active] != pass) return;
  int d[PEPO_MAXLEG];
  load_dims(it.x, ival, d);
  const int nl = it.x.nlegs;
  const int F = 4 * (nl > 0 ? d[nl - 1] : 1);
  long long K = 1;
  for (int i = 0; i + 1 < nl; ++i) K *= d[i];
  const int S = exact_splits(K);
  if (acct && blockIdx.x == 0 && threadIdx.x == 0) {
    atomicAdd(&acct[0], (double)K * F * (F + 1.0));
    atomicAdd(&acct[1], (double)K * F * sizeof(float));
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < F * F; e += gridDim.x * blockDim.x) {
    const int fi = e / F, fj = e - fi * F;
    if (fi > fj) continue;
    double sum = 0.0;
    for (int s = 0; s < S; ++s) sum += it.partial[(long long)s * F * F + e];
    it.out[(long long)fi * it.ldo + fj] = sum;
    it.out[(long long)fj * it.ldo + fi] = sum;
  }
}

cudaError_t launch_gram_exact(const GramRowsItem* items, int n_items, int fmax, int pass, void* const* ptrs,
                              const int* ival, double* acct, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  k_col_scale<<<dim3(1, n_items), 256, 0, s>>>(items, pass, 0, ptrs, ival);
  k_col_scale<<<dim3(64, n_items), 256, 0, s>>>(items, pass, 1, ptrs, ival);
  const size_t smem = sizeof(float) * (4 * GX_RUN * GX_T + 2 * GX_T * GX_T);
  cudaError_t e = cudaFuncSetAttribute(k_gram_exact, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int nt = ceil_div(fmax, GX_T);
  k_gram_exact<<<dim3(nt * (nt + 1) / 2 * kExactSplits, 1, n_items), 256, smem, s>>>(items, pass, ptrs, ival);
  int gx = ceil_div(fmax * fmax, 256);
  if (gx > 256) gx = 256;
  k_gram_exact_reduce<<<dim3(gx, n_items), 256, 0, s>>>(items, pass, ival, acct);
  return cudaGetLastError();
}

// ================================================================ reconstruct
// out[r, (c', p')] = sum_{(c,p)} in[r, (c,p)] W[(c,p), (c',p')], stored in the
// permuted output layout.
//
// FP64: 64 x 64 output tiles, K streamed 16 at a time.
constexpr int RC_T = 64;
constexpr int RC_BK = 16;

template <typename T>
__global__ void __launch_bounds__(256)
k_reconstruct(const ReconItem* __restrict__ items, void* const* ptrs, const int* __restrict__ ival) {
  const ReconItem it = items[blockIdx.y];
  int d[PEPO_MAXLEG];
  load_dims(it.in, ival, d);
  const int nl = it.in.nlegs;
  const int cut = nl - 1;
  const int n = 4 * d[cut];
  const int chin = ival[it.new_dim];
  const int np = 4 * chin;
  long long R = 1;
  for (int i = 0; i < cut; ++i) R *= d[i];
  // output strides per input leg
  int od[PEPO_MAXLEG];
  for (int i = 0; i < nl; ++i) od[i] = (i == cut) ? chin : d[i];
  long long ostride_in[PEPO_MAXLEG];   // stride of input leg i in the output
  {
    long long st = 4;
    for (int kk = nl - 1; kk >= 0; --kk) {
      int li = it.out_perm[kk];
      ostride_in[li] = st;
      st *= od[li];
    }
  }
  long long rstride[PEPO_MAXLEG];      // stride of env leg i inside the row index
  {
    long long st = 1;
    for (int i = cut - 1; i >= 0; --i) { rstride[i] = st; st *= d[i]; }
  }
  const int nct = ceil_div(np, RC_T);
  const long long nrt = (R + RC_T - 1) / RC_T;
  const long long units = nrt * nct;
  const T* __restrict__ in = static_cast<const T*>(ptrs[it.in.ref]);
  T* __restrict__ out = static_cast<T*>(ptrs[it.out_ref]);
  __shared__ __align__(16) T As[RC_BK][RC_T + 4];
  __shared__ __align__(16) T Ws[RC_BK][RC_T];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  for (long long u = blockIdx.x; u < units; u += gridDim.x) {
    const long long rt = u / nct;
    const int ct = (int)(u - rt * nct);
    const long long r0 = rt * RC_T;
    const int c0 = ct * RC_T;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    for (int kb = 0; kb < n; kb += RC_BK) {
      for (int e = threadIdx.x; e < RC_BK * RC_T; e += blockDim.x) {
        // A tile: rows r0.., k kb..  (read rows contiguously along k)
        int rr = e / RC_BK, kk = e - rr * RC_BK;
        long long r = r0 + rr;
        int kx = kb + kk;
        As[kk][rr] = (r < R && kx < n) ? in[r * n + kx] : T(0);
        int kk2 = e / RC_T, cc = e - kk2 * RC_T;
        int ky = kb + kk2, cy = c0 + cc;
        Ws[kk2][cc] = (ky < n && cy < np) ? (T)it.W[(long long)ky * it.ldw + cy] : T(0);
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < RC_BK; ++kk) {
        T xa[4], yb[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) xa[a] = As[kk][ty * 4 + a];
#pragma unroll
        for (int b = 0; b < 4; ++b) yb[b] = Ws[kk][tx * 4 + b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] = fma(xa[a], yb[b], acc[a][b]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      long long r = r0 + ty * 4 + a;
      if (r >= R) continue;
      long long base = 0, rem = r;
      for (int i = 0; i < cut; ++i) {
        long long idx = rem / rstride[i];
        rem -= idx * rstride[i];
        base += idx * ostride_in[i];
      }
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        int c = c0 + tx * 4 + b;
        if (c >= np) continue;
        int cn = c >> 2, p = c & 3;
        out[base + cn * ostride_in[cut] + p] = acc[a][b];
      }
    }
  }
}

// FP32: 256 x 64 tiles.  The tiles of all items, column by column, are one sequence
// that is shared out evenly among the CTAs the chip holds (the items of a wave
// differ by chi^2 in rows).  A CTA keeps its 64 columns of W, rounded to FP32 once,
// in shared memory (W is FP64, and a conversion takes the FP64 unit) and goes
// through row tiles with them; the rows arrive as they lie, 16 values of K at a
// time, as asynchronous 16-byte copies three stages deep and across tiles.  A
// thread holds 8 x 8 entries: per four values of K, 8 + 8 16-byte shared loads
// (8 rows 80 bytes apart, or 4 neighbouring quads: no bank conflicts) for 256
// multiply-adds.  The rows are numbered with the output's innermost row leg
// fastest, so that 8 lanes store 16-byte neighbours.  The sum over K runs in order.
// Bound: FP32 ALU.  Class of a 4x4 chi = 48 layer, 64 x 64 tiles with scalar
// loads -> these tiles -> one even sequence: 12.4 -> 5.6 -> 3.6 ms.
constexpr int R3_ROWS = 256, R3_COLS = 64, R3_K = 16, R3_PITCH = R3_K + 4, R3_STAGES = 3;

struct R3Plan {
  int n, chin;
  unsigned R;
  unsigned e1, e2;                                     // row = (a0, a1, a2): extents of a1, a2
  unsigned rs[3];                                      // strides among the input's rows
  long long os[3], ocut;                               // and in the output; the new cut leg's
  const float* in;
  float* out;
  const double* W;
  int ldw;
};
__device__ __noinline__ void r3_plan(const ReconItem& it, const int* ival, void* const* ptrs, R3Plan& p) {
  p.in = static_cast<const float*>(ptrs[it.in.ref]);
  p.out = static_cast<float*>(ptrs[it.out_ref]);
  p.W = it.W;
  p.ldw = it.ldw;
  const int nl = it.in.nlegs, cut = nl - 1;
  p.chin = ival[it.new_dim];
  p.n = 4 * ival[it.in.dim[cut]];
  // output stride of a leg: 4 x the extents of the legs that follow it in out_perm
  long long os[PEPO_MAXLEG] = {0, 0, 0, 0};
  unsigned dd[PEPO_MAXLEG] = {1, 1, 1, 1}, rs[PEPO_MAXLEG] = {0, 0, 0, 0};
  long long st = 4;
  for (int kk = nl - 1; kk >= 0; --kk) {
    const int l = it.out_perm[kk];
    os[l] = st;
    dd[l] = l == cut ? p.chin : ival[it.in.dim[l]];
    st *= dd[l];
  }
  p.R = 1;
  for (int l = cut - 1; l >= 0; --l) { rs[l] = p.R; p.R *= dd[l]; }
  // the (up to three) row legs, the output's innermost one last
  const int inner = it.out_perm[nl - 1];
  int leg[3] = {-1, -1, -1}, at = 2;
  if (inner != cut && cut > 0) leg[at--] = inner;
  for (int l = cut - 1; l >= 0 && at >= 0; --l)
    if (l != inner) leg[at--] = l;
  for (int i = 0; i < 3; ++i) {
    p.rs[i] = leg[i] >= 0 ? rs[leg[i]] : 0;
    p.os[i] = leg[i] >= 0 ? os[leg[i]] : 0;
  }
  p.e1 = leg[1] >= 0 ? dd[leg[1]] : 1;
  p.e2 = leg[2] >= 0 ? dd[leg[2]] : 1;
  p.ocut = os[cut];
}

// Row tiles of one column tile from tile `at` of the item, at most `most`; returns how many.
__device__ __noinline__ unsigned r3_tiles(const R3Plan& pl, float* r3_sh, unsigned at, unsigned most) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ty = 8 * (warp >> 1) + (lane & 7), tx = 4 * (warp & 1) + (lane >> 3);
  const int n = pl.n, np = 4 * pl.chin;
  const unsigned R = pl.R, nrt = (R + R3_ROWS - 1) / R3_ROWS;
  const float* __restrict__ in = pl.in;
  float* __restrict__ out = pl.out;
  float* Ws = r3_sh;                                   // [n][64]
  float* As = r3_sh + (size_t)n * R3_COLS;             // stages of [256][pitch]
  const unsigned nch = (unsigned)ceil_div(n, R3_K);
  const int ct = (int)(at / nrt);
  const unsigned first = at - ct * nrt, tiles = min(nrt - first, most), total = tiles * nch;
  for (int e = tid; e < n * R3_COLS; e += 256) {
    const int c = ct * R3_COLS + (e & (R3_COLS - 1));
    Ws[e] = c < np ? (float)pl.W[(long long)(e / R3_COLS) * pl.ldw + c] : 0.f;
  }
  // load cursor: this thread copies quad tid % 4 of the rows tid / 4 + 64 u
  unsigned li = 0, lch = 0, ltile = first;
  unsigned src[4];                                   // row of the input (~0: none)
  auto load = [&]() {
    if (li < total) {
      if (lch == 0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const unsigned r = ltile * R3_ROWS + (tid >> 2) + 64 * u;
          const unsigned q = r / pl.e2, a2 = r - q * pl.e2, a0 = q / pl.e1, a1 = q - a0 * pl.e1;
          src[u] = r < R ? a0 * pl.rs[0] + a1 * pl.rs[1] + a2 * pl.rs[2] : ~0u;
        }
      }
      const int k = lch * R3_K + 4 * (tid & 3);
      float* dst = As + (li % R3_STAGES) * (R3_ROWS * R3_PITCH) + (tid >> 2) * R3_PITCH + 4 * (tid & 3);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool live = src[u] != ~0u && k < n;
        copy_quad(dst + 64 * u * R3_PITCH, live ? in + (long long)src[u] * n + k : in, live);
      }
      if (++lch == nch) { lch = 0; ++ltile; }
      ++li;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int st = 0; st < R3_STAGES - 1; ++st) load();
  float acc[8][2][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 8; ++b) acc[a][b >> 2][b & 3] = 0.f;
  unsigned tile = first, ch = 0;
  for (unsigned m = 0; m < total; ++m) {
    asm volatile("cp.async.wait_group %0;" ::"n"(R3_STAGES - 2) : "memory");
    __syncthreads();                                 // this chunk is in, the one before is consumed
    load();
    const float* as = As + (m % R3_STAGES) * (R3_ROWS * R3_PITCH) + ty * R3_PITCH;
    const float* ws = Ws + (size_t)ch * (R3_K * R3_COLS) + 4 * tx;
    const int kn = min(R3_K, n - (int)ch * R3_K);    // a multiple of 4
    for (int k = 0; k < kn; k += 4) {
      float x[8][4];
#pragma unroll
      for (int a = 0; a < 8; ++a)
        *reinterpret_cast<float4*>(x[a]) = *reinterpret_cast<const float4*>(as + 32 * a * R3_PITCH + k);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        float w[2][4];
        *reinterpret_cast<float4*>(w[0]) = *reinterpret_cast<const float4*>(ws + (k + kk) * R3_COLS);
        *reinterpret_cast<float4*>(w[1]) = *reinterpret_cast<const float4*>(ws + (k + kk) * R3_COLS + 32);
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int b = 0; b < 8; ++b) acc[a][b >> 2][b & 3] = fmaf(x[a][kk], w[b >> 2][b & 3], acc[a][b >> 2][b & 3]);
      }
    }
    if (++ch < nch) continue;
    ch = 0;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      const unsigned r = tile * R3_ROWS + ty + 32 * a;
      if (r < R) {
        const unsigned q = r / pl.e2, a2 = r - q * pl.e2, a0 = q / pl.e1, a1 = q - a0 * pl.e1;
        float* dst = out + a0 * pl.os[0] + a1 * pl.os[1] + a2 * pl.os[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const int cn = ct * (R3_COLS / 4) + tx + 8 * b;
          if (cn < pl.chin) *reinterpret_cast<float4*>(dst + cn * pl.ocut) = *reinterpret_cast<const float4*>(acc[a][b]);
        }
      }
#pragma unroll
      for (int b = 0; b < 8; ++b) acc[a][b >> 2][b & 3] = 0.f;
    }
    ++tile;
  }
  return tiles;
}

__global__ void __launch_bounds__(256, 2)
k_reconstruct32(const ReconItem* __restrict__ items, int n_items, void* const* ptrs, const int* __restrict__ ival) {
  __shared__ R3Plan pl;
  __shared__ unsigned toff[kMaxItems + 1];
  extern __shared__ __align__(16) float r3_sh[];
  tile_prefix(toff, n_items, [&](int i) {
    const ReconItem& it = items[i];
    const int cut = it.in.nlegs - 1;
    unsigned R = 1;
    for (int l = 0; l < cut; ++l) R *= ival[it.in.dim[l]];
    return (R + R3_ROWS - 1) / R3_ROWS * ceil_div(4 * ival[it.new_dim], R3_COLS);
  });
  const unsigned nt = toff[n_items], share = nt / gridDim.x, more = nt - share * gridDim.x;
  unsigned t = blockIdx.x * share + min(blockIdx.x, more);
  const unsigned t1 = t + share + (blockIdx.x < more ? 1 : 0);
  if (t >= t1) return;
  int item = tile_item(toff, n_items, t);
  while (t < t1) {
    while (toff[item + 1] <= t) ++item;
    __syncthreads();                                   // the plan and the columns before are consumed
    if (threadIdx.x == 0) r3_plan(items[item], ival, ptrs, pl);
    __syncthreads();
    t += r3_tiles(pl, r3_sh, t - toff[item], t1 - t);
  }
}

template <typename T>
cudaError_t launch_reconstruct(const ReconItem* items, int n_items, int chimax, void* const* ptrs, const int* ival,
                               cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  const int nmax = 4 * chimax;
  if constexpr (sizeof(T) == 4) {
    const size_t smem = sizeof(float) * ((size_t)nmax * R3_COLS + (size_t)R3_STAGES * R3_ROWS * R3_PITCH);
    cudaError_t e = cudaFuncSetAttribute(k_reconstruct32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    for (int i0 = 0; i0 < n_items; i0 += kMaxItems)
      k_reconstruct32<<<2 * 152, 256, smem, s>>>(items + i0, std::min(kMaxItems, n_items - i0), ptrs, ival);
  } else {
    const long long rows = (long long)chimax * chimax * chimax;
    const long long tiles = (rows + RC_T - 1) / RC_T * ceil_div(nmax, RC_T);
    const int gx = (int)std::max<long long>(4, std::min<long long>(tiles, 2 * 152 * 4 / n_items + 1));
    k_reconstruct<T><<<dim3(gx, n_items), 256, 0, s>>>(items, ptrs, ival);
  }
  return cudaGetLastError();
}

// ========================================================= vector contraction
// Sum of products x v, x of the storage type, v FP64.  FP32 storage: v as two FP32
// parts and a two-float sum (12 FP32 operations a product, ~2^-45 of the sum's
// terms; an FP64 multiply-add and the conversion take 128 issue slots here).  C_proj of
// stored states is within 7e-15 of 64 bits either way.
template <typename T> struct VecSum;
template <> struct VecSum<double> {
  double s = 0.0;
  __device__ void add(double x, double v) { s = fma(x, v, s); }
  __device__ void merge(int o) { s += __shfl_xor_sync(0xffffffffu, s, o); }
  __device__ double value() const { return s; }
  static __device__ double split(double v) { return v; }
  using V = double;
};
template <> struct VecSum<float> : TwoFloat {
  using V = float2;
  static __device__ float2 split(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
  }
  __device__ void add(float x, float2 v) {
    take_product(x, v.x);
    c = fmaf(x, v.y, c);
  }
  __device__ void merge(int o) {
    const float p = __shfl_xor_sync(0xffffffffu, s, o), q = __shfl_xor_sync(0xffffffffu, c, o);
    take(p);
    c += q;
  }
};

// One pass over the pinned slice feeds both first contractions: lanes hold the
// columns j3, so a row's product with v_last is a warp sum and the products with
// v_prev accumulate per lane.  A block shares the rows of one o when there are
// 32 or more, else each of its warps takes an o of its own.  Bound: HBM (every
// 32-byte sector of the site tensor holds two pinned values); separate passes
// read the tensor twice and kept the FP64 pipe busy for 4 slots a value.
// A row's sum goes to FP64 with up to 31 others, a lane each: one at a time the three
// FP64 operations of it cost as much as the row's load.
// Class of the correlator of a 4x4, chi = 64 grid (11 passes): 7.2 -> 4.3 -> 3.8 ms; of a
// batch of nine small instances 53 -> 5.5 ms (blocks per item by their number).
template <typename T>
__global__ void __launch_bounds__(256)
k_vec_pair(const VecPairItem* __restrict__ items, void* const* ptrs, const int* __restrict__ ival) {
  using A = VecSum<T>;
  const VecPairItem it = items[blockIdx.y];
  int d[PEPO_MAXLEG];
#pragma unroll
  for (int k = 0; k < PEPO_MAXLEG; ++k) d[k] = (k < it.ndims) ? ival[it.dim[k]] : 1;
  long long O = 1;
  int J2 = 1, J3 = 1;
#pragma unroll
  for (int k = 0; k < PEPO_MAXLEG; ++k) {
    if (k == it.ndims - 1) J3 = d[k];
    else if (k == it.ndims - 2) J2 = d[k];
    else if (k < it.ndims) O *= d[k];
  }
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool share = J2 >= 32;
  if ((share ? (long long)blockIdx.x : (long long)blockIdx.x * 8) >= O) return;
  __shared__ typename A::V vl[128], vp[128];
  __shared__ double part[8][128];
  for (int i = tid; i < J3; i += 256) vl[i] = A::split(it.v_last[i]);
  for (int i = tid; i < J2; i += 256) vp[i] = A::split(it.v_prev[i]);
  __syncthreads();
  const T* site = static_cast<const T*>(ptrs[it.in_ref]) + it.pin;
  const long long step = share ? gridDim.x : (long long)gridDim.x * 8;
  for (long long o = share ? blockIdx.x : (long long)blockIdx.x * 8 + w; o < O; o += step) {
    const T* base = site + o * J2 * J3 * 4;
    A col[4], kept;                                    // lane r keeps the sum of the warp's row r mod 32
    int r = 0;
    const int first = share ? w : 0, by = share ? 8 : 1;
    for (int j2 = first; j2 < J2; j2 += by) {
      T x[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j3 = lane + 32 * c;
        x[c] = j3 < J3 ? __ldg(base + ((long long)j2 * J3 + j3) * 4) : T(0);
      }
      A row;
      const typename A::V q = vp[j2];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j3 = lane + 32 * c;
        if (j3 < J3) {
          row.add(x[c], vl[j3]);
          col[c].add(x[c], q);
        }
      }
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) row.merge(m);
      if (lane == (r & 31)) kept = row;
      ++r;
      if ((r & 31) == 0 || j2 + by >= J2) {            // up to 32 sums go to FP64 at once
        const int at = first + ((r - 1) / 32 * 32 + lane) * by;
        if (lane <= ((r - 1) & 31)) it.out_prev[o * J2 + at] = kept.value();
      }
    }
    if (share) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (lane + 32 * c < J3) part[w][lane + 32 * c] = col[c].value();
      __syncthreads();
      for (int j = tid; j < J3; j += 256) {
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < 8; ++i) t += part[i][j];
        it.out_last[o * J3 + j] = t;
      }
      __syncthreads();
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (lane + 32 * c < J3) it.out_last[o * J3 + lane + 32 * c] = col[c].value();
    }
  }
}

// blocks per item: about 16 per SM in all, few per item when a batch has many
static int vec_blocks(int n_items) { return max(4, min(256, ceil_div(16 * 152, n_items))); }

template <typename T>
cudaError_t launch_vec_pair(const VecPairItem* items, int n_items, void* const* ptrs, const int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  k_vec_pair<T><<<dim3(vec_blocks(n_items), n_items), 256, 0, s>>>(items, ptrs, ival);
  return cudaGetLastError();
}

template <typename T>
__global__ void k_vec_contract(const VecItem* __restrict__ items, void* const* ptrs,
                               const int* __restrict__ ival) {
  const VecItem it = items[blockIdx.y];
  int d[PEPO_MAXLEG];
#pragma unroll
  for (int k = 0; k < PEPO_MAXLEG; ++k) d[k] = (k < it.ndims) ? ival[it.dim[k]] : 1;
  const int k = it.leg;
  if (k < 0) {  // no contraction: the pinned slice of a one-leg site
    const T* site = static_cast<const T*>(ptrs[it.in_ref]);
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < d[0]; e += gridDim.x * blockDim.x)
      it.out[e] = (double)site[e * 4 + it.pin];
    return;
  }
  unsigned O = 1, Q = 1;
  int J = 1;
#pragma unroll
  for (int i = 0; i < PEPO_MAXLEG; ++i) {
    if (i == k) J = d[i];
    else if (i < k) O *= d[i];
    else if (i < it.ndims) Q *= d[i];
  }
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < O * Q; e += gridDim.x * blockDim.x) {
    const unsigned o = e / Q, q = e - o * Q;
    const double* x = it.in_d + (long long)o * J * Q + q;
    double sum = 0.0;
#pragma unroll 4
    for (int j = 0; j < J; ++j) sum = fma(x[(long long)j * Q], it.v[j], sum);
    it.out[e] = sum;
  }
}

template <typename T>
cudaError_t launch_vec_contract(const VecItem* items, int n_items, void* const* ptrs, const int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  k_vec_contract<T><<<dim3(min(32, vec_blocks(n_items)), n_items), 256, 0, s>>>(items, ptrs, ival);
  return cudaGetLastError();
}

// ============================================================ instantiations
#define PEPO_INST(T)                                                                              \
  template cudaError_t launch_copy<T>(const TView*, const int*, int, int, void* const*,           \
                                      const int*, cudaStream_t);                                  \
  template cudaError_t launch_gram_rows<T>(const GramRowsItem*, int, int, int, int, void* const*, \
                                           const int*, cudaStream_t);                             \
  template cudaError_t launch_reconstruct<T>(const ReconItem*, int, int, void* const*,            \
                                             const int*, cudaStream_t);                           \
  template cudaError_t launch_vec_contract<T>(const VecItem*, int, void* const*, const int*,      \
                                              cudaStream_t);                                      \
  template cudaError_t launch_vec_pair<T>(const VecPairItem*, int, void* const*, const int*,      \
                                          cudaStream_t);
PEPO_INST(float)
PEPO_INST(double)

}  // namespace pepo
