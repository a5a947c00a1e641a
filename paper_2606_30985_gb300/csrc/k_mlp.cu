// Learned BP warm start: feature rows, a 3-layer MLP (forward, backward,
// Adam) and the message writer.  The paper has no learned part; in this
// extension of the method, per directed bond e and Schmidt
// index k the MLP predicts y = log diag(M_e)[k] of the converged double-layer
// message (Eq. 13 fixed point) in the bond's Schmidt basis, and damped BP then
// starts from M_e = diag(exp(y)) / sum exp(y).
//
// Precision: weights and activations are rounded to BF16 (round to nearest
// even) at the layer inputs, every product is accumulated in FP32, gradients
// and the Adam state are FP32 on an FP32 master copy of the weights.
// GEMMs have width 256 and K <= 256 except the weight gradients, whose K is the
// row count; they run as 128 x 128 register-tiled SIMT tiles.
#include <cuda_bf16.h>

#include "kernels.h"
#include "mlp.h"

namespace pepo {

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float x) {
  const float cdf = 0.5f * (1.f + erff(x * 0.70710678118654752f));
  const float pdf = 0.39894228040143268f * expf(-0.5f * x * x);
  return cdf + x * pdf;
}

// ---------------------------------------------------------------- SIMT GEMM
// C[m, n] = sum_k A[m, k] B[k, n].  AT = 0: A row-major [M x K]; 1: A stored
// [K x M] (a weight gradient's activations).  BT = 0: B row-major [K x N]; 1: B
// stored [N x K].  Every load is 16 bytes along the stored row.  epi: 0 = store
// C; 1 = store z = C + bias and a = bf16(gelu(z)); 2 = store C * gelu'(zref).
// grid.z splits K: split s writes its partial sum at C + s M ldc.
//
// 128 x 128 tiles, 8 x 8 entries a thread, the next 16-deep slice in registers
// while one is multiplied.  Bound: FP32 ALU.  One 10x10, chi = 100 layer
// (36000 rows): the three 256 x 256 x rows products are 1.4e10 FLOP, 0.18 ms at
// the FP32 peak; a weight gradient's K = rows is split so that it fills the
// chip (16 tiles of 64 x 64 ran over all rows one after another before).  The
// whole training step on those rows: 14.1 -> 0.68 ms.
struct GemmArgs {
  const float* A; int lda;
  const float* B; int ldb;
  float* C; int ldc;
  const float* bias;
  float* act;            // epi 1: rounded activation, leading dimension ldc
  const float* zref;     // epi 2: pre-activation the derivative is taken at
  int M, N, K;           // N a multiple of 4; K too unless AT; M too when AT
  int epi;
};

constexpr int MG_T = 128, MG_BK = 16;

template <int AT, int BT>
__global__ void __launch_bounds__(256) k_mlp_gemm(GemmArgs g) {
  __shared__ __align__(16) float As[MG_BK][MG_T + 4];
  __shared__ __align__(16) float Bs[MG_BK][MG_T + 4];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * MG_T, n0 = blockIdx.x * MG_T;
  const int kc = (g.K + gridDim.z - 1) / gridDim.z;
  const int k0 = blockIdx.z * kc, k1 = min(g.K, k0 + kc);
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 ra[2], rb[2];
  auto load = [&](int k) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = tid + 256 * u;
      if (AT) {              // 16 rows (k) of 32 quads (m)
        const int kk = k + (e >> 5), m = m0 + 4 * (e & 31);
        ra[u] = kk < k1 && m < g.M ? *reinterpret_cast<const float4*>(g.A + (long long)kk * g.lda + m) : zero;
      } else {               // 128 rows (m) of 4 quads (k)
        const int m = m0 + (e >> 2), kk = k + 4 * (e & 3);
        ra[u] = m < g.M && kk < k1 ? *reinterpret_cast<const float4*>(g.A + (long long)m * g.lda + kk) : zero;
      }
      if (BT) {
        const int n = n0 + (e >> 2), kk = k + 4 * (e & 3);
        rb[u] = n < g.N && kk < k1 ? *reinterpret_cast<const float4*>(g.B + (long long)n * g.ldb + kk) : zero;
      } else {
        const int kk = k + (e >> 5), n = n0 + 4 * (e & 31);
        rb[u] = kk < k1 && n < g.N ? *reinterpret_cast<const float4*>(g.B + (long long)kk * g.ldb + n) : zero;
      }
    }
  };
  auto store = [&]() {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = tid + 256 * u;
      if (AT) {
        *reinterpret_cast<float4*>(&As[e >> 5][4 * (e & 31)]) = ra[u];
      } else {
        const int m = e >> 2, kk = 4 * (e & 3);
        As[kk][m] = ra[u].x; As[kk + 1][m] = ra[u].y; As[kk + 2][m] = ra[u].z; As[kk + 3][m] = ra[u].w;
      }
      if (BT) {
        const int n = e >> 2, kk = 4 * (e & 3);
        Bs[kk][n] = rb[u].x; Bs[kk + 1][n] = rb[u].y; Bs[kk + 2][n] = rb[u].z; Bs[kk + 3][n] = rb[u].w;
      } else {
        *reinterpret_cast<float4*>(&Bs[e >> 5][4 * (e & 31)]) = rb[u];
      }
    }
  };
  float acc[8][8] = {};
  load(k0);
  for (int k = k0; k < k1; k += MG_BK) {
    store();
    __syncthreads();
    if (k + MG_BK < k1) load(k + MG_BK);
#pragma unroll
    for (int kk = 0; kk < MG_BK; ++kk) {
      float av[8], bv[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {   // rows / columns 4 t .. 4 t + 3 and 64 further
        *reinterpret_cast<float4*>(av + 4 * h) = *reinterpret_cast<const float4*>(&As[kk][64 * h + 4 * ty]);
        *reinterpret_cast<float4*>(bv + 4 * h) = *reinterpret_cast<const float4*>(&Bs[kk][64 * h + 4 * tx]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
  float* C = g.C + (long long)blockIdx.z * g.M * g.ldc;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + 64 * (i >> 2) + 4 * ty + (i & 3);
    if (m >= g.M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int n = n0 + 64 * h + 4 * tx;
      if (n >= g.N) continue;
      const long long o = (long long)m * g.ldc + n;
      float v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = acc[i][4 * h + q];
      if (g.epi == 1) {
        float t[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) { v[q] += g.bias[n + q]; t[q] = bf16r(gelu_f(v[q])); }
        *reinterpret_cast<float4*>(g.act + o) = make_float4(t[0], t[1], t[2], t[3]);
      } else if (g.epi == 2) {
        const float4 z = *reinterpret_cast<const float4*>(g.zref + o);
        v[0] *= gelu_grad_f(z.x); v[1] *= gelu_grad_f(z.y); v[2] *= gelu_grad_f(z.z); v[3] *= gelu_grad_f(z.w);
      }
      *reinterpret_cast<float4*>(C + o) = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

template <int AT, int BT>
static cudaError_t gemm(const GemmArgs& g, int splits, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  dim3 grid((g.N + MG_T - 1) / MG_T, (g.M + MG_T - 1) / MG_T, splits);
  k_mlp_gemm<AT, BT><<<grid, 256, 0, s>>>(g);
  return cudaGetLastError();
}

// out[i] = sum of `parts` partial vectors of length n
__global__ void k_sum_parts(const float* __restrict__ part, int parts, int n, float* __restrict__ out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int p = 0; p < parts; ++p) s += part[(long long)p * n + i];
    out[i] = s;
  }
}

// y[r] = a[r, :] . w + b: one warp per row
__global__ void __launch_bounds__(256)
k_row_dot(const float* __restrict__ a, const float* __restrict__ w, const float* __restrict__ b, int rows,
          float* __restrict__ y) {
  constexpr int W = PEPO_WS_WIDTH;
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (r >= rows) return;
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < W; k += 128) {
    const float4 x = *reinterpret_cast<const float4*>(a + (long long)r * W + k + 4 * lane);
    const float4 v = *reinterpret_cast<const float4*>(w + k + 4 * lane);
    s = fmaf(x.x, v.x, s); s = fmaf(x.y, v.y, s); s = fmaf(x.z, v.z, s); s = fmaf(x.w, v.w, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) y[r] = s + b[0];
}

// Backward of the output layer in one pass over z2 and a2, one thread per
// column and a chunk of rows per block: d2 = dy W3^T gelu'(z2), and the
// chunk's part of dW3 = a2^T dy and db2 = column sums of d2 (out: [chunk][2][W]).
// Memory-bound; a single block per 128 columns summed all rows before.
__global__ void __launch_bounds__(PEPO_WS_WIDTH)
k_out_backward(const float* __restrict__ z2, const float* __restrict__ a2, const float* __restrict__ dy,
               const float* __restrict__ w3, int rows, int chunk, float* __restrict__ d2, float* __restrict__ dw3,
               float* __restrict__ db2, long long stride) {
  constexpr int W = PEPO_WS_WIDTH;
  const int c = threadIdx.x;
  const int r0 = blockIdx.x * chunk, r1 = min(rows, r0 + chunk);
  const float w = w3[c];
  float s3 = 0.f, s2 = 0.f;
#pragma unroll 4
  for (int r = r0; r < r1; ++r) {
    const long long o = (long long)r * W + c;
    const float e = dy[r];
    const float d = (e * w) * gelu_grad_f(z2[o]);
    d2[o] = d;
    s2 += d;
    s3 = fmaf(a2[o], e, s3);
  }
  dw3[blockIdx.x * stride + c] = s3;
  db2[blockIdx.x * stride + c] = s2;
}

// The chunk's part of dW1 = x^T d1 and db1 = column sums of d1 (out: [chunk][13][W])
__global__ void __launch_bounds__(PEPO_WS_WIDTH)
k_in_backward(const float* __restrict__ x, const float* __restrict__ d1, int rows, int chunk, float* __restrict__ out) {
  constexpr int W = PEPO_WS_WIDTH, F = PEPO_WS_FEATURES;
  const int c = threadIdx.x;
  const int r0 = blockIdx.x * chunk, r1 = min(rows, r0 + chunk);
  float acc[F + 1] = {};
#pragma unroll 2
  for (int r = r0; r < r1; ++r) {
    const float d = d1[(long long)r * W + c];
#pragma unroll
    for (int f = 0; f < F; ++f) acc[f] = fmaf(x[(long long)r * F + f], d, acc[f]);
    acc[F] += d;
  }
  float* o = out + (long long)blockIdx.x * (F + 1) * W;
#pragma unroll
  for (int f = 0; f <= F; ++f) o[f * W + c] = acc[f];
}

__global__ void k_round(const float* in, float* out, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = bf16r(in[i]);
}

// dy = 2 / n (y - t), the loss and db3 = sum dy (one block: deterministic sums)
__global__ void __launch_bounds__(1024) k_mse(const float* y, const float* t, int n, float* dy, float* loss, float* db3) {
  __shared__ float red[1024], rb[1024];
  float s = 0.f, sd = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float d = y[i] - t[i];
    const float e = 2.f * d / (float)n;
    dy[i] = e;
    s += d * d;
    sd += e;
  }
  red[threadIdx.x] = s;
  rb[threadIdx.x] = sd;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) { red[threadIdx.x] += red[threadIdx.x + o]; rb[threadIdx.x] += rb[threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { *loss = red[0] / (float)n; *db3 = rb[0]; }
}

__global__ void k_adam(float* p, float* m, float* v, const float* g, long long n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ------------------------------------------------------------------ features
// One block per directed bond (b, dir).  Rows of bond b start at
// sum_{b' < b} 2 chi_b' + dir chi_b.
__device__ double entropy_fraction(const double* lam, int chi) {
  if (chi < 2) return 0.0;
  double s = 0.0;
  for (int k = 0; k < chi; ++k) {
    const double p = lam[k] * lam[k];
    if (p > 0.0) s -= p * log(p);
  }
  return s / log((double)chi);
}

__global__ void k_ws_features(const WsGeom* __restrict__ geom, int nb, const int* __restrict__ chi,
                              const double* __restrict__ lam, int ldl, float t, float h, float J, float* X,
                              int max_rows) {
  const int db = blockIdx.x;            // directed bond 2 b + dir
  const int b = db >> 1, dir = db & 1;
  __shared__ long long off;
  __shared__ float sf[4];
  if (threadIdx.x == 0) {
    long long o = 0;
    for (int e = 0; e < b; ++e) o += 2LL * chi[e];
    off = o + (long long)dir * chi[b];
  }
  const WsGeom G = geom[db];
  if (threadIdx.x < 4) {
    const int e = threadIdx.x == 0 ? b : (threadIdx.x - 1 < G.n_other ? G.other[threadIdx.x - 1] : -1);
    sf[threadIdx.x] = e >= 0 ? (float)entropy_fraction(lam + (long long)e * ldl, chi[e]) : 0.f;
  }
  __syncthreads();
  float mean_nb = 0.f, max_nb = 0.f;
  for (int i = 0; i < G.n_other; ++i) { mean_nb += sf[1 + i]; max_nb = fmaxf(max_nb, sf[1 + i]); }
  if (G.n_other > 0) mean_nb /= (float)G.n_other;
  const int c = chi[b];
  for (int k = threadIdx.x; k < c; k += blockDim.x) {
    const long long r = off + k;
    if (r >= max_rows) continue;
    float* x = X + r * PEPO_WS_FEATURES;
    const double lk = fmax(lam[(long long)b * ldl + k], 1e-30);
    x[0] = (float)log(lk);
    x[1] = (float)k / (float)c;
    x[2] = sf[0];
    x[3] = G.deg_src * 0.25f;
    x[4] = G.deg_dst * 0.25f;
    x[5] = G.dist_src;
    x[6] = G.dist_dst;
    x[7] = t;
    x[8] = h;
    x[9] = J;
    x[10] = mean_nb;
    x[11] = max_nb;
  }
}

// targets: y = log M_e[k, k] of the current messages (after BP)
__global__ void k_ws_targets(int nb, const int* __restrict__ chi, const double* __restrict__ msg, int ldm,
                             float* out, int max_rows) {
  const int db = blockIdx.x;
  const int b = db >> 1, dir = db & 1;
  __shared__ long long off;
  if (threadIdx.x == 0) {
    long long o = 0;
    for (int e = 0; e < b; ++e) o += 2LL * chi[e];
    off = o + (long long)dir * chi[b];
  }
  __syncthreads();
  const int c = chi[b];
  const double* M = msg + (long long)db * ldm * ldm;
  for (int k = threadIdx.x; k < c; k += blockDim.x) {
    const long long r = off + k;
    if (r < max_rows) out[r] = (float)log(fmax(M[(long long)k * ldm + k], 1e-300));
  }
}

// messages <- diag((1 - gamma) d / sum d + gamma exp(y) / sum exp(y)), zero
// elsewhere; d = diagonal of the current message (the diag(lambda) written by
// the bond updates), exp(y) max-shifted
__global__ void k_ws_apply(int nb, const int* __restrict__ chi, const float* __restrict__ y, double* msg, int ldm,
                           float gamma) {
  const int db = blockIdx.x;
  const int b = db >> 1, dir = db & 1;
  __shared__ long long off;
  __shared__ double red[256], red2[256];
  __shared__ float ymax;
  if (threadIdx.x == 0) {
    long long o = 0;
    for (int e = 0; e < b; ++e) o += 2LL * chi[e];
    off = o + (long long)dir * chi[b];
  }
  __syncthreads();
  const int c = chi[b];
  double* M = msg + (long long)db * ldm * ldm;
  if (threadIdx.x == 0) {
    float m = -INFINITY;
    for (int k = 0; k < c; ++k) m = fmaxf(m, y[off + k]);
    ymax = m;
  }
  __syncthreads();
  double s = 0.0, sd = 0.0;
  for (int k = threadIdx.x; k < c; k += blockDim.x) {
    s += exp((double)(y[off + k] - ymax));
    sd += M[(long long)k * ldm + k];
  }
  red[threadIdx.x] = s;
  red2[threadIdx.x] = sd;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) { red[threadIdx.x] += red[threadIdx.x + o]; red2[threadIdx.x] += red2[threadIdx.x + o]; }
    __syncthreads();
  }
  const double tot = red[0], totd = red2[0];
  // diagonal first (read before the overwrite), then the rest
  double dk[8];
  int nk = 0;
  for (int k = threadIdx.x; k < c && nk < 8; k += blockDim.x) dk[nk++] = M[(long long)k * ldm + k];
  __syncthreads();
  nk = 0;
  for (int k = threadIdx.x; k < c && nk < 8; k += blockDim.x) {
    const double plain = totd > 0.0 ? dk[nk] / totd : 0.0;
    dk[nk++] = (1.0 - gamma) * plain + gamma * exp((double)(y[off + k] - ymax)) / tot;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < ldm * ldm; e += blockDim.x) {
    const int i = e / ldm, j = e - i * ldm;
    if (i != j || i >= c) M[e] = 0.0;
  }
  nk = 0;
  for (int k = threadIdx.x; k < c && nk < 8; k += blockDim.x) M[(long long)k * ldm + k] = dk[nk++];
}

// ------------------------------------------------------------------ launchers
cudaError_t launch_ws_features(const WsGeom* geom, int nb, const int* chi, const double* lam, int ldl, float t,
                               float h, float J, float* X, int max_rows, cudaStream_t s) {
  if (nb == 0) return cudaSuccess;
  k_ws_features<<<2 * nb, 128, 0, s>>>(geom, nb, chi, lam, ldl, t, h, J, X, max_rows);
  return cudaGetLastError();
}
cudaError_t launch_ws_targets(int nb, const int* chi, const double* msg, int ldm, float* out, int max_rows,
                              cudaStream_t s) {
  if (nb == 0) return cudaSuccess;
  k_ws_targets<<<2 * nb, 128, 0, s>>>(nb, chi, msg, ldm, out, max_rows);
  return cudaGetLastError();
}
cudaError_t launch_ws_apply(int nb, const int* chi, const float* y, double* msg, int ldm, float gamma,
                            cudaStream_t s) {
  if (nb == 0) return cudaSuccess;
  k_ws_apply<<<2 * nb, 256, 0, s>>>(nb, chi, y, msg, ldm, gamma);
  return cudaGetLastError();
}

// Parameter offsets in the flat vector: W1 [NF x W], b1 [W], W2 [W x W], b2 [W], W3 [W], b3 [1]
struct MlpOff {
  long long W1, b1, W2, b2, W3, b3, n;
};
static MlpOff mlp_off() {
  MlpOff o;
  const long long F = PEPO_WS_FEATURES, W = PEPO_WS_WIDTH;
  o.W1 = 0;
  o.b1 = o.W1 + F * W;
  o.W2 = o.b1 + W;
  o.b2 = o.W2 + W * W;
  o.W3 = o.b2 + W;
  o.b3 = o.W3 + W;
  o.n = o.b3 + 1;
  return o;
}

long long mlp_num_params() { return mlp_off().n; }

size_t mlp_layout(char* base, int max_rows, MlpBuffers* B) {
  const MlpOff o = mlp_off();
  const size_t W = PEPO_WS_WIDTH, F = PEPO_WS_FEATURES, R = (size_t)max_rows;
  size_t off = 0;
  auto take = [&](size_t n) {
    off = (off + 63) / 64 * 64;
    float* p = base ? reinterpret_cast<float*>(base + off) : nullptr;
    off += n * sizeof(float);
    return p;
  };
  B->p = take(o.n);
  B->m = take(o.n);
  B->v = take(o.n);
  B->g = take(o.n);
  B->pr = take(o.n);
  B->x = take(R * F);
  B->z1 = take(R * W);
  B->a1 = take(R * W);
  B->z2 = take(R * W);
  B->a2 = take(R * W);
  B->y = take(R);
  B->dy = take(R);
  B->d2 = take(R * W);
  B->d1 = take(R * W);
  B->loss = take(4);
  return off + 64;
}

// forward pass on the rounded weights; activations kept for backward
cudaError_t mlp_forward(const MlpBuffers& B, const float* X, int rows, float* y_out, cudaStream_t s) {
  const MlpOff o = mlp_off();
  const int W = PEPO_WS_WIDTH, F = PEPO_WS_FEATURES;
  k_round<<<256, 256, 0, s>>>(B.p, B.pr, o.n);
  k_round<<<256, 256, 0, s>>>(X, B.x, (long long)rows * F);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  GemmArgs g{};
  g.A = B.x; g.lda = F;
  g.B = B.pr + o.W1; g.ldb = W;
  g.C = B.z1; g.ldc = W; g.bias = B.p + o.b1; g.act = B.a1;
  g.M = rows; g.N = W; g.K = F; g.epi = 1;
  if ((e = gemm<0, 0>(g, 1, s)) != cudaSuccess) return e;
  g.A = B.a1; g.lda = W;
  g.B = B.pr + o.W2;
  g.C = B.z2; g.bias = B.p + o.b2; g.act = B.a2; g.K = W;
  if ((e = gemm<0, 0>(g, 1, s)) != cudaSuccess) return e;
  k_row_dot<<<(rows + 7) / 8, 256, 0, s>>>(B.a2, B.pr + o.W3, B.p + o.b3, rows, y_out ? y_out : B.y);
  return cudaGetLastError();
}

// forward + backward of the mean squared error; gradient into B.g, loss into B.loss[0]
cudaError_t mlp_gradient(const MlpBuffers& B, const float* X, const float* t, int rows, cudaStream_t s) {
  const MlpOff o = mlp_off();
  const int W = PEPO_WS_WIDTH, F = PEPO_WS_FEATURES;
  cudaError_t e = mlp_forward(B, X, rows, B.y, s);
  if (e != cudaSuccess) return e;
  k_mse<<<1, 1024, 0, s>>>(B.y, t, rows, B.dy, B.loss, B.g + o.b3);
  // Row chunks of the column sums: about two blocks per SM, at least 32 rows.
  // Partial sums go to activation buffers that nothing needs any more (d1 before
  // it is formed; z2 and a2 after d2 is), which hold them for every row count:
  // a single chunk writes the gradient itself.
  const int chunk = rows / 304 > 32 ? (rows + 303) / 304 : 32;
  const int nch = (rows + chunk - 1) / chunk;
  // dz2 = (dy W3^T) * gelu'(z2), dW3 = a2^T dy, db2 = colsum dz2
  if (nch == 1) {
    k_out_backward<<<1, W, 0, s>>>(B.z2, B.a2, B.dy, B.pr + o.W3, rows, chunk, B.d2, B.g + o.W3, B.g + o.b2, 0);
  } else {
    k_out_backward<<<nch, W, 0, s>>>(B.z2, B.a2, B.dy, B.pr + o.W3, rows, chunk, B.d2, B.d1, B.d1 + (long long)nch * W, W);
    k_sum_parts<<<1, W, 0, s>>>(B.d1, nch, W, B.g + o.W3);
    k_sum_parts<<<1, W, 0, s>>>(B.d1 + (long long)nch * W, nch, W, B.g + o.b2);
  }
  // dW2 = a1^T dz2, K = rows split so that 4 tiles x splits fill the chip, at least 256 rows each
  const int splits = rows / 256 < 1 ? 1 : (rows / 256 < 76 ? rows / 256 : 76);
  GemmArgs g{};
  g.A = B.a1; g.lda = W;                     // stored [rows x W]
  g.B = B.d2; g.ldb = W;
  g.C = splits == 1 ? B.g + o.W2 : B.a2; g.ldc = W; g.M = W; g.N = W; g.K = rows; g.epi = 0;
  if ((e = gemm<1, 0>(g, splits, s)) != cudaSuccess) return e;
  if (splits > 1) k_sum_parts<<<W * W / 256, 256, 0, s>>>(B.a2, splits, W * W, B.g + o.W2);
  // dz1 = (dz2 W2^T) * gelu'(z1)
  GemmArgs d{};
  d.A = B.d2; d.lda = W;
  d.B = B.pr + o.W2; d.ldb = W;              // stored [W x W], used transposed
  d.C = B.d1; d.ldc = W; d.zref = B.z1; d.M = rows; d.N = W; d.K = W; d.epi = 2;
  if ((e = gemm<0, 1>(d, 1, s)) != cudaSuccess) return e;
  // dW1 = x^T dz1, db1 = colsum dz1 (neighbours in the parameter vector)
  if (nch == 1) {
    k_in_backward<<<1, W, 0, s>>>(B.x, B.d1, rows, chunk, B.g + o.W1);
  } else {
    k_in_backward<<<nch, W, 0, s>>>(B.x, B.d1, rows, chunk, B.z2);
    k_sum_parts<<<F + 1, W, 0, s>>>(B.z2, nch, (F + 1) * W, B.g + o.W1);
  }
  return cudaGetLastError();
}

cudaError_t mlp_adam(const MlpBuffers& B, int t, float lr, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
  k_adam<<<128, 256, 0, s>>>(B.p, B.m, B.v, B.g, mlp_off().n, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace pepo
