// SIMT contractions of the BP and bond-update hot loop (FP32 and FP64 modes).
//
//   k_leg_contract  out[o, i, q] = sum_j A[i, j] in[o, j, q] on one layout leg
//                   (absorbing a message factor or eigenbasis into a site
//                   tensor: Sec. 2.5 step 1 and the products of Eq. 13)
//   k_gram_leg      out[i, i'] = sum_{o, q} X[o, i, q] X[o, i', q]: a site tensor
//                   contracted with itself over every index but one leg, the
//                   Pauli leg traced (one double-layer message, Eq. 13; the
//                   message weights are carried by the rotated tensor)
//
// Both are GEMMs with one short dimension (chi <= 128); tiles are chosen from
// the live bond dimension on the device.  FP32 storage accumulates the Gram's
// long sums in FP32 runs of 256 terms that a two-float sum takes.
#include <algorithm>
#include <type_traits>

#include "kernels.h"

namespace pepo {

constexpr int GL_FLUSH = 256;   // FP32 terms per run of a Gram

__device__ inline void load_dims4(const TView& v, const int* ival, int* d) {
#pragma unroll
  for (int k = 0; k < PEPO_MAXLEG; ++k) d[k] = (k < v.nlegs) ? ival[v.dim[k]] : 1;
}

// ============================================================ leg contraction
// out[o, i, q] = sum_j A[i, j] in[o, j, q], i.e. a (Jout x J) matrix times the J x C
// matrix of the columns c = (o, q), q fastest and contiguous.  FP32: the grid is what
// the chip holds; the tiles of TC columns of all items, in one sequence, are
// shared out evenly (items differ by chi^2 between a corner and the bulk).  A CTA
// keeps its item's A transposed in shared memory; rows of `in` arrive eight at a
// time as asynchronous 16-byte copies (a unit of 16 bytes never leaves its o),
// three stages deep and across tiles, and a thread holds MI outputs of NU
// units.  TI = MI x (NT / column threads) is chosen from the live Jout, so a small
// bond does not pay for the rows of a large tile.  The sum over j runs in order.
//
// Bound: FP32 ALU at chi = 48 (12 FLOP per byte), HBM below, launch and latency below
// chi = 20.  Class of a case, 64 / 128-row tiles -> whole tiles loaded, then
// multiplied, a fixed grid per item -> these: BP legs of a 4x4 chi = 48 layer 72 -> 24 ->
// 21 ms, of nine 4x4 instances 76 -> 14 -> 6.5 ms.
// FP64 is bound by its pipe, two multiply-adds per clock and SM, so its tiles
// are small (64 threads, one unit each) and a small site still spreads over
// many SMs: at chi = 8 a tile of 512 columns took one SM 8 us (class 6.0 -> 3.5 ms).
template <typename T> struct LegBlock;
template <> struct LegBlock<float> { static constexpr int NT = 256, CTAS = 2; };
template <> struct LegBlock<double> { static constexpr int NT = 64, CTAS = 8; };
constexpr int kLegRows = 8, kLegStages = 3;
template <typename T, int MI, int TI>
struct LegCfg {
  static constexpr int U = 16 / (int)sizeof(T);
  static constexpr int IG = TI / MI;                   // thread groups over the outputs
  static constexpr int CG = LegBlock<T>::NT / IG;      // threads over the columns
  static constexpr int NU = sizeof(T) == 4 && TI > 16 ? 2 : 1;   // units per thread
  static constexpr int TU = CG * NU;                   // units of a tile
  static constexpr int TC = TU * U;                    // columns
  static constexpr int PITCH = TC + U;                 // values between staged rows (one unit off the banks)
};

// units of a tile and rows of A for a live Jout
template <typename T>
__host__ __device__ inline int leg_ti(int Jout) {
  if (sizeof(T) == 4 && (Jout > 16 && Jout <= 24 || Jout > 32 && Jout <= 48 || Jout > 64 && Jout <= 96)) return Jout <= 24 ? 24 : Jout <= 48 ? 48 : 96;
  return Jout <= 8 ? 8 : Jout <= 16 ? 16 : Jout <= 32 ? 32 : Jout <= 64 ? 64 : 128;
}
template <typename T>
__host__ __device__ inline int leg_tu(int ti) {
  return ti == 8 ? LegCfg<T, 4, 8>::TU : ti == 16 ? LegCfg<T, 8, 16>::TU : ti <= 32 ? LegCfg<T, 8, 32>::TU
       : ti <= 64 ? LegCfg<T, 8, 64>::TU : LegCfg<T, 8, 128>::TU;   // 24, 48, 96: as many groups, six rows each
}

// tiles lo .. hi - 1 of an item
template <typename T, int MI, int TI>
__device__ void leg_tiles(const T* __restrict__ in, T* __restrict__ out, const double* __restrict__ A, int lda, int J,
                          int Jout, unsigned O, unsigned QU, unsigned char* sh, unsigned lo, unsigned hi) {
  using C = LegCfg<T, MI, TI>;
  constexpr int U = C::U, CG = C::CG, NU = C::NU, PITCH = C::PITCH, TU = C::TU, NT = LegBlock<T>::NT;
  const int tid = threadIdx.x;
  const int cg = tid % CG, ig = tid / CG;
  const long long Q = (long long)QU * U;
  const unsigned cols = O * QU;                        // columns in units
  T* At = reinterpret_cast<T*>(sh);                    // [J][TI]
  T* Bs = At + (size_t)J * TI;                 // [stage][row][PITCH]
  const unsigned nch = J > kLegRows ? (J + kLegRows - 1) / kLegRows : 1;
  const unsigned total = (hi - lo) * nch;
  // load cursor.  Threads run along the columns, the groups share the rows; on the
  // innermost leg (QU = 1: a column's rows are 16 bytes apart) eight threads
  // run along the rows instead, so that they read 128 consecutive bytes.
  unsigned ltile = lo, lch = 0, li = 0;
  const uint4* in4 = reinterpret_cast<const uint4*>(in);
  unsigned src[NU];                                    // first unit of the thread's column (~0: none)
  auto load = [&]() {
    if (li < total) {
      const int j0 = lch * kLegRows, jn = min(kLegRows, J - j0);
      T* dst = Bs + (size_t)(li % kLegStages) * (kLegRows * PITCH);
      auto copy = [&](int j, int c, unsigned at, bool live) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(dst + j * PITCH + c * U)),
                     "l"(in4 + (live ? at : 0u)), "r"(live ? 16 : 0)
                     : "memory");
      };
      if (QU == 1) {
        const int j = tid & (kLegRows - 1);
        if (j < jn)
#pragma unroll
          for (int c = tid / kLegRows; c < TU; c += NT / kLegRows) {
            const unsigned o = ltile * TU + c;
            copy(j, c, o * (unsigned)J + j0 + j, o < cols);
          }
      } else {
        if (lch == 0) {
#pragma unroll
          for (int u = 0; u < NU; ++u) {
            const unsigned c = ltile * TU + u * CG + cg;
            const unsigned o = c / QU;
            src[u] = c < cols ? o * (J - 1) * QU + c : ~0u;   // a tensor has below 2^30 units
          }
        }
        for (int j = ig; j < jn; j += C::IG)
#pragma unroll
          for (int u = 0; u < NU; ++u) copy(j, u * CG + cg, src[u] + (j0 + j) * QU, src[u] != ~0u);
      }
      if (++lch == nch) { lch = 0; ++ltile; }
      ++li;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  __syncthreads();                                     // the item before is consumed
#pragma unroll
  for (int st = 0; st < kLegStages - 1; ++st) load();
  for (int e = tid; e < J * TI; e += NT) {
    const int i = e / J, j = e - i * J;
    const T x = i < Jout ? (T)A[(long long)i * lda + j] : T(0);
    At[j * TI + i] = x;
  }
  T acc[MI][NU][U];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int u = 0; u < NU; ++u)
#pragma unroll
      for (int x = 0; x < U; ++x) acc[i][u][x] = T(0);
  unsigned tile = lo, ch = 0;
  for (unsigned n = 0; n < total; ++n) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kLegStages - 2) : "memory");
    __syncthreads();                                   // this chunk is in, the one before is consumed
    load();
    const T* b0 = Bs + (size_t)(n % kLegStages) * (kLegRows * PITCH) + cg * U;
    const T* a0 = At + (size_t)ch * (kLegRows * TI) + ig * MI;
    auto step = [&](int j) {
      T b[NU][U];
#pragma unroll
      for (int u = 0; u < NU; ++u)
        *reinterpret_cast<uint4*>(b[u]) = *reinterpret_cast<const uint4*>(b0 + j * PITCH + u * CG * U);
      {
        T a[MI];
#pragma unroll
        for (int i = 0; i < MI; i += MI % U ? U / 2 : U) {
          if constexpr (MI % U != 0) *reinterpret_cast<uint2*>(a + i) = *reinterpret_cast<const uint2*>(a0 + j * TI + i);
          else *reinterpret_cast<uint4*>(a + i) = *reinterpret_cast<const uint4*>(a0 + j * TI + i);
        }
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
          for (int u = 0; u < NU; ++u)
#pragma unroll
            for (int x = 0; x < U; ++x) acc[i][u][x] = fma(a[i], b[u][x], acc[i][u][x]);
      }
    };
    const int jn = min(kLegRows, J - (int)ch * kLegRows);
#pragma unroll 2
    for (int j = 0; j < jn; ++j) step(j);
    if (++ch < nch) continue;
    ch = 0;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      const unsigned c = tile * TU + u * CG + cg;
      if (c < cols) {
        const unsigned o = c / QU, q = c - o * QU;
        T* dst = out + (long long)o * Jout * Q + (long long)q * U;
#pragma unroll
        for (int i = 0; i < MI; ++i) {
          const int io = ig * MI + i;
          if (io < Jout) *reinterpret_cast<uint4*>(dst + (long long)io * Q) = *reinterpret_cast<const uint4*>(acc[i][u]);
        }
      }
    }
    ++tile;
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
      for (int u = 0; u < NU; ++u)
#pragma unroll
        for (int x = 0; x < U; ++x) acc[i][u][x] = T(0);
  }
}

template <typename T>
__global__ void __launch_bounds__(LegBlock<T>::NT, LegBlock<T>::CTAS)
k_leg_contract(const LegItem* __restrict__ items, int n_items, void* const* ptrs, const int* __restrict__ ival) {
  extern __shared__ __align__(16) unsigned char lc_sh[];
  __shared__ unsigned toff[kMaxItems + 1];          // tiles before each item
  auto extents = [&](const LegItem& it, int& J, unsigned& O, unsigned& QU) {
    int d[PEPO_MAXLEG];
    load_dims4(it.in, ival, d);
    unsigned Q = 4;
    J = 1;
    O = 1;
#pragma unroll
    for (int i = 0; i < PEPO_MAXLEG; ++i) {
      if (i == it.leg) J = d[i];
      else if (i < it.leg) O *= d[i];
      else Q *= d[i];                                  // legs beyond nlegs have size 1
    }
    QU = Q / (16 / sizeof(T));
  };
  auto run = [&](const LegItem& it, int J, int Jout, unsigned O, unsigned QU, unsigned lo, unsigned hi) {
    const int lda = it.lda;
    const double* A = it.A;
    const T* in = static_cast<const T*>(ptrs[it.in.ref]);
    T* out = static_cast<T*>(ptrs[it.out_ref]);
    switch (leg_ti<T>(Jout)) {
      case 8: leg_tiles<T, 4, 8>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi); break;
      case 16: leg_tiles<T, 8, 16>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi); break;
      case 32: leg_tiles<T, 8, 32>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi); break;
      case 64: leg_tiles<T, 8, 64>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi); break;
      case 128: leg_tiles<T, 8, 128>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi); break;
      default:
        if constexpr (sizeof(T) == 4) {
          if (Jout <= 24) leg_tiles<T, 6, 24>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi);
          else if (Jout <= 48) leg_tiles<T, 6, 48>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi);
          else leg_tiles<T, 6, 96>(in, out, A, lda, J, Jout, O, QU, lc_sh, lo, hi);
        }
    }
  };
  if constexpr (sizeof(T) == 8) {                      // a grid row per item
    const LegItem& it = items[blockIdx.y];
    int J;
    unsigned O, QU;
    extents(it, J, O, QU);
    const int Jout = ival[it.out_dim];
    const unsigned tu = leg_tu<T>(leg_ti<T>(Jout)), nt = (O * QU + tu - 1) / tu;
    const unsigned per = nt / gridDim.x, more = nt - per * gridDim.x;
    const unsigned lo = blockIdx.x * per + min(blockIdx.x, more), hi = lo + per + (blockIdx.x < more ? 1 : 0);
    if (lo < hi) run(it, J, Jout, O, QU, lo, hi);
  } else {
    tile_prefix(toff, n_items, [&](int i) {
      int J;
      unsigned O, QU;
      extents(items[i], J, O, QU);
      const unsigned tu = leg_tu<T>(leg_ti<T>(ival[items[i].out_dim]));
      return (O * QU + tu - 1) / tu;
    });
    const unsigned nt = toff[n_items], per = nt / gridDim.x, more = nt - per * gridDim.x;
    unsigned t = blockIdx.x * per + min(blockIdx.x, more);
    const unsigned t1 = t + per + (blockIdx.x < more ? 1 : 0);
    int item = tile_item(toff, n_items, t);
    while (t < t1) {
      while (toff[item + 1] <= t) ++item;
      const LegItem& it = items[item];
      int J;
      unsigned O, QU;
      extents(it, J, O, QU);
      const unsigned lo = t - toff[item], hi = min(t1, toff[item + 1]) - toff[item];
      run(it, J, ival[it.out_dim], O, QU, lo, hi);
      t += hi - lo;
    }
  }
}

template <typename T>
cudaError_t launch_leg_contract(const LegItem* items, int n_items, int chimax, void* const* ptrs, const int* ival,
                                cudaStream_t s) {
  size_t smem = 0;                                     // A and the stages of every tile that a live bond may take
  for (int ti = 8; ti <= 128 && ti < 2 * chimax + 8; ti *= 2)
    smem = std::max(smem, sizeof(T) * (size_t)chimax * ti + (size_t)kLegStages * kLegRows * (leg_tu<T>(ti) + 1) * 16);
  cudaError_t e = cudaFuncSetAttribute(k_leg_contract<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  for (int i0 = 0; i0 < n_items; i0 += kMaxItems) {
    const int n = std::min(kMaxItems, n_items - i0);
    // FP64: a row of the grid per item (a small launch is all latency, and the
    // shared sequence has more of it: 8.1 -> 11.4 us at chi = 8)
    const dim3 grid = sizeof(T) == 8 ? dim3(std::max(8, 8 * 152 / n), n) : dim3(152 * LegBlock<T>::CTAS);
    k_leg_contract<T><<<grid, LegBlock<T>::NT, smem, s>>>(items + i0, n, ptrs, ival);
  }
  return cudaGetLastError();
}

// ============================================================ Gram (free leg)
// out[i, i'] = sum over the flattened (o, q) of X[o, i, q] X[o, i', q]: X is F rows
// of O Q values, contiguous in q.  One CTA takes one split of the summed range
// of one item.  Chunks of KCU 16-byte units per row (a unit never leaves its
// o: Q is a multiple of 4) are copied asynchronously as they lie, three stages
// deep; rows are KCU + 1 units apart, an odd number, so the 8 threads of a
// phase read 8 different banks groups.  TX x TX threads share a tile of MT TX
// rows, thread (ty, tx) holding the entries (ty + TX a, tx + TX b) with a <= b
// only: the Gram is symmetric, and this drops 44 % of the products for the
// largest tile without a divergent branch.  The 256 / TX^2 groups of threads
// take different units of a chunk, so a small F keeps the whole block busy;
// the tile is chosen from the live F (8, 16, 24, 32, 48, 64, 96, 128), not from
// chi_max.  Their sums are laid side by side and added by one thread per entry: with
// the groups adding one after another, a warp's FP64 operations (64 clocks each)
// in 16 turns took longer than the products of a small split.  FP32 storage sums runs
// of 256 terms in FP32 and the runs in a two-float sum (which is within 1e-16 of the
// rows' norms of an FP64 sum of them); FP64 sums directly.
//
// Bound: shared memory (a 16-byte load of a warp takes 4 clocks of the SM, 2 where
// neighbouring lanes share it, and MT + MT of them feed 2 MT (MT + 1) products), so up
// to F = 32 the threads of a group are 4 x 4 with as many entries each as that
// takes: 24 clocks of loads per unit at F = 32 instead of 48 with 8 x 8 threads;
// or the FP64 pipe.  Class of a case, before -> now: chi = 8 FP64 (107 launches)
// 143 -> 1.8 ms, 4x4 chi = 12 FP64 154 -> 1.7 ms, 4x4 chi = 48 FP32 82 -> 25 ms.  The
// 64 x 64 (128 x 128) tile it replaces did 64 x 64 products for an 8 x 8 Gram and
// stored every chunk with 32-way bank conflicts.
constexpr int kGlStages = 3;

template <typename T, int MT, int TX>
struct GlCfg {
  static constexpr int U = 16 / (int)sizeof(T);        // values per 16-byte unit
  static constexpr int TL = MT * TX;
  static constexpr int G = 256 / (TX * TX);            // groups sharing a chunk
  static constexpr int U0 = sizeof(T) == 4 ? 16 : 8;
  static constexpr int KCU = (U0 / 4) * G > U0 ? (U0 / 4) * G : U0;   // units per row and chunk
  static constexpr int PITCH = (KCU + 1) * U;          // values between rows
  static constexpr size_t kStage = sizeof(T) * (size_t)TL * PITCH;
  using V = std::conditional_t<sizeof(T) == 4, float2, double>;   // a group's sum of an entry
  static constexpr size_t kRed = G > 1 ? sizeof(V) * (size_t)G * TL * TL : 0;
  static constexpr size_t kSmem = kGlStages * kStage > kRed ? kGlStages * kStage : kRed;
};

template <typename T, int MT, int TX>
__device__ void gram_tile(const T* __restrict__ X, long long O, long long Q, int F, int s, int S, double* __restrict__ P,
                          unsigned char* sh) {
  using C = GlCfg<T, MT, TX>;
  constexpr int U = C::U, KCU = C::KCU, G = C::G, TL = C::TL, PITCH = C::PITCH;
  constexpr bool kF32 = sizeof(T) == 4;
  T* buf = reinterpret_cast<T*>(sh);
  const int tid = threadIdx.x;
  const int g = tid / (TX * TX), t = tid % (TX * TX), tx = t % TX, ty = t / TX;
  const unsigned QU = (unsigned)(Q / U);               // units per (o, row)
  const unsigned NU = (unsigned)(O * Q / U);           // units of the summed range
  const unsigned NC = (NU + KCU - 1) / KCU;
  const unsigned c0 = (unsigned)((unsigned long long)NC * s / S), c1 = (unsigned)((unsigned long long)NC * (s + 1) / S);
  const int lu = tid % KCU, lf0 = tid / KCU;           // this thread's unit of a chunk, first row
  constexpr int LR = 256 / KCU;                        // rows per pass
  // rows F .. TL - 1 are zero in every stage
  for (int st = 0; st < kGlStages; ++st)
    for (int e = tid; e < (TL - F) * PITCH; e += 256) buf[st * (TL * PITCH) + F * PITCH + e] = T(0);
  auto load = [&](unsigned c, int st) {
    if (c < c1) {
      const unsigned u = c * KCU + lu;
      const bool live = u < NU;
      const unsigned o = live ? u / QU : 0u, q = live ? u - o * QU : 0u;
      const T* src = X + ((long long)o * F) * Q + (long long)q * U;
      T* dst = buf + st * (TL * PITCH) + lu * U;
      for (int f = lf0; f < F; f += LR)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(dst + f * PITCH)),
                     "l"(live ? src + (long long)f * Q : X), "r"(live ? 16 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  T acc[MT][MT];
  float hi[MT][MT], lo[MT][MT];                        // FP32: two-float sum of the runs
#pragma unroll
  for (int a = 0; a < MT; ++a)
#pragma unroll
    for (int b = 0; b < MT; ++b) { acc[a][b] = T(0); hi[a][b] = lo[a][b] = 0.f; }
  auto flush = [&]() {
    if constexpr (kF32) {
#pragma unroll
      for (int a = 0; a < MT; ++a)
#pragma unroll
        for (int b = a; b < MT; ++b) {
          const float v = acc[a][b], w = hi[a][b] + v, z = w - hi[a][b];
          lo[a][b] += (hi[a][b] - (w - z)) + (v - z);
          hi[a][b] = w;
          acc[a][b] = 0.f;
        }
    }
  };
  __syncthreads();
#pragma unroll
  for (int st = 0; st < kGlStages - 1; ++st) load(c0 + st, st);
  int st = 0, run = 0;
  for (unsigned c = c0; c < c1; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kGlStages - 2) : "memory");
    __syncthreads();                                   // chunk c is in, chunk c - 1 is consumed
    load(c + kGlStages - 1, st == 0 ? kGlStages - 1 : st - 1);
    const T* xs = buf + st * (TL * PITCH);
#pragma unroll
    for (int k = 0; k < KCU / G; ++k) {
      const int u = g * (KCU / G) + k;
      T av[MT][U];
#pragma unroll
      for (int a = 0; a < MT; ++a) {
        const uint4 x = *reinterpret_cast<const uint4*>(xs + (ty + TX * a) * PITCH + u * U);
        *reinterpret_cast<uint4*>(av[a]) = x;
      }
#pragma unroll
      for (int b = 0; b < MT; ++b) {
        T bv[U];
        *reinterpret_cast<uint4*>(bv) = *reinterpret_cast<const uint4*>(xs + (tx + TX * b) * PITCH + u * U);
#pragma unroll
        for (int i = 0; i < U; ++i)
#pragma unroll
          for (int a = 0; a <= b; ++a) acc[a][b] = fma(av[a][i], bv[i], acc[a][b]);
      }
    }
    if constexpr (kF32) {
      run += KCU / G * U;
      if (run >= GL_FLUSH) { flush(); run = 0; }
    }
    if (++st == kGlStages) st = 0;
  }
  flush();
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if constexpr (G > 1) {
    // sum of the groups' values, one thread per entry of the blocks a <= b, the groups in
    // order; the other triangle is a mirror
    using V = typename C::V;
    V* red = reinterpret_cast<V*>(sh);
    __syncthreads();
#pragma unroll
    for (int a = 0; a < MT; ++a)
#pragma unroll
      for (int b = a; b < MT; ++b) {
        V* r = red + (g * TL + ty + TX * a) * TL + tx + TX * b;
        if constexpr (kF32) *r = make_float2(hi[a][b], lo[a][b]);
        else *r = acc[a][b];
      }
    __syncthreads();
    for (int e = tid; e < MT * (MT + 1) / 2 * TX * TX; e += 256) {
      int b = e / (TX * TX), a = 0;
      while (b >= MT - a) { b -= MT - a; ++a; }        // block (a, a + b)
      const int in = e % (TX * TX), i = TX * a + in / TX, j = TX * (a + b) + in % TX;
      if (i >= F || j >= F) continue;
      double z = 0.0;
      TwoFloat t;
#pragma unroll
      for (int gg = 0; gg < G; ++gg) {
        const V v = red[(gg * TL + i) * TL + j];
        if constexpr (kF32) {
          t.take(v.x);
          t.c += v.y;
        } else {
          z += v;
        }
      }
      if constexpr (kF32) z = t.value();
      P[(long long)i * F + j] = z;
      if (b > 0) P[(long long)j * F + i] = z;
    }
  } else {
#pragma unroll
    for (int a = 0; a < MT; ++a)
#pragma unroll
      for (int b = a; b < MT; ++b) {
        const int i = ty + TX * a, j = tx + TX * b;
        if (i < F && j < F) {
          double v;
          if constexpr (kF32) v = (double)hi[a][b] + (double)lo[a][b];
          else v = acc[a][b];
          P[(long long)i * F + j] = v;
          if (a != b) P[(long long)j * F + i] = v;
        }
      }
  }
}

// Bands of F, a launch of its own for each that chi_max can reach, so that the
// small tiles do not carry the large ones' registers (two blocks per SM up to
// F = 24 and for 33 .. 48): blocks of the other bands return.
constexpr int kGramBands[] = {0, 24, 32, 48, 64, 128};
template <typename T, int BAND>
__global__ void __launch_bounds__(256, BAND == 0 || BAND == 2 ? 2 : 1)
k_gram_leg(const GramLegItem* __restrict__ items, int splits_max, void* const* ptrs, const int* __restrict__ ival) {
  const GramLegItem it = items[blockIdx.y];
  int d[PEPO_MAXLEG];
  load_dims4(it.x, ival, d);
  const int k = it.leg;
  int F = 1;
  long long O = 1, Q = 4;
#pragma unroll
  for (int i = 0; i < PEPO_MAXLEG; ++i) {
    if (i == k) F = d[i];
    else if (i < k) O *= d[i];
    else Q *= d[i];                                    // legs beyond nlegs have size 1
  }
  constexpr int kAbove = BAND == 0 ? -1 : kGramBands[BAND], kUpTo = kGramBands[BAND + 1];
  if (F <= kAbove || F > kUpTo) return;
  const int S = gram_leg_splits_k(O * Q, splits_max, gram_leg_rows_simt(sizeof(T)));
  extern __shared__ __align__(16) unsigned char gl_sh[];
  const T* X = static_cast<const T*>(ptrs[it.x.ref]);
  for (int s = blockIdx.x; s < S; s += gridDim.x) {
    double* P = it.partial + (long long)s * F * F;
    if constexpr (BAND == 0) {
      if (F <= 8) gram_tile<T, 2, 4>(X, O, Q, F, s, S, P, gl_sh);
      else if (F <= 16) gram_tile<T, 4, 4>(X, O, Q, F, s, S, P, gl_sh);
      else gram_tile<T, 6, 4>(X, O, Q, F, s, S, P, gl_sh);
    } else if constexpr (BAND == 1) {
      gram_tile<T, 8, 4>(X, O, Q, F, s, S, P, gl_sh);
    } else if constexpr (BAND == 2) {
      gram_tile<T, 6, 8>(X, O, Q, F, s, S, P, gl_sh);
    } else if constexpr (BAND == 3) {
      gram_tile<T, 8, 8>(X, O, Q, F, s, S, P, gl_sh);
    } else {
      if (F <= 96) gram_tile<T, 6, 16>(X, O, Q, F, s, S, P, gl_sh);
      else gram_tile<T, 8, 16>(X, O, Q, F, s, S, P, gl_sh);
    }
    __syncthreads();                                   // the shared memory is reused
  }
}

template <typename T, int BAND>
size_t gram_leg_smem() {
  if (BAND == 0) return std::max(std::max(GlCfg<T, 2, 4>::kSmem, GlCfg<T, 4, 4>::kSmem), GlCfg<T, 6, 4>::kSmem);
  if (BAND == 1) return GlCfg<T, 8, 4>::kSmem;
  if (BAND == 2) return GlCfg<T, 6, 8>::kSmem;
  if (BAND == 3) return GlCfg<T, 8, 8>::kSmem;
  return std::max(GlCfg<T, 6, 16>::kSmem, GlCfg<T, 8, 16>::kSmem);
}

__global__ void k_gram_leg_reduce(const GramLegItem* __restrict__ items, int splits_max, int rows, int sym,
                                  const int* __restrict__ ival) {
  const GramLegItem it = items[blockIdx.y];
  int d[PEPO_MAXLEG];
  load_dims4(it.x, ival, d);
  const int k = it.leg;
  const int F = d[k];
  long long O = 1, Q = 4;
  for (int i = 0; i < k; ++i) O *= d[i];
  for (int i = k + 1; i < it.x.nlegs; ++i) Q *= d[i];
  const int S = gram_leg_splits_k(O * Q, splits_max, rows);
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < F * F; e += gridDim.x * blockDim.x) {
    int fi = e / F, fj = e - fi * F;
    double sum = 0.0;
    for (int s = 0; s < S; ++s) sum += it.partial[(long long)s * F * F + e];
    if (sym) {
      double st = 0.0;
      for (int s = 0; s < S; ++s) st += it.partial[(long long)s * F * F + (long long)fj * F + fi];
      sum = 0.5 * (sum + st);
    }
    it.out[(long long)fi * it.ldo + fj] = sum;
  }
}

template <typename T, int BAND>
static cudaError_t launch_gram_band(const GramLegItem* items, int n_items, int splits_max, void* const* ptrs,
                                    const int* ival, cudaStream_t s) {
  const size_t smem = gram_leg_smem<T, BAND>();
  cudaError_t e = cudaFuncSetAttribute(k_gram_leg<T, BAND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // about 16 blocks per SM in all; a block takes several splits of its item when
  // there are many items (a batch), so that few of its blocks find nothing to do
  const int gx = std::min(splits_max, std::max(8, ceil_div(16 * 152, n_items)));
  k_gram_leg<T, BAND><<<dim3(gx, n_items), 256, smem, s>>>(items, splits_max, ptrs, ival);
  return cudaGetLastError();
}

int gram_leg_launches(int chimax) {
  int n = 1;
  while (n < 5 && chimax > kGramBands[n]) ++n;
  return n;
}

template <typename T>
cudaError_t launch_gram_leg(const GramLegItem* items, int n_items, int splits_max, int chimax,
                            void* const* ptrs, const int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  cudaError_t e = launch_gram_band<T, 0>(items, n_items, splits_max, ptrs, ival, s);
  const int bands = gram_leg_launches(chimax);
  if (e == cudaSuccess && bands > 1) e = launch_gram_band<T, 1>(items, n_items, splits_max, ptrs, ival, s);
  if (e == cudaSuccess && bands > 2) e = launch_gram_band<T, 2>(items, n_items, splits_max, ptrs, ival, s);
  if (e == cudaSuccess && bands > 3) e = launch_gram_band<T, 3>(items, n_items, splits_max, ptrs, ival, s);
  if (e == cudaSuccess && bands > 4) e = launch_gram_band<T, 4>(items, n_items, splits_max, ptrs, ival, s);
  return e;
}

cudaError_t launch_gram_leg_reduce(const GramLegItem* items, int n_items, int chimax,
                                   int splits_max, int rows, int sym, const int* ival, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  int gx = ceil_div(chimax * chimax, 256);
  k_gram_leg_reduce<<<dim3(gx, n_items), 256, 0, s>>>(items, splits_max, rows, sym, ival);
  return cudaGetLastError();
}

// ==================================================================== permute
// Canonical site layout -> stored layout (or back): out[perm position] = in[i].
// perm[k] = canonical leg index at layout position k; dims in canonical order.
template <typename T>
__global__ void k_permute(const T* __restrict__ in, T* __restrict__ out, int nlegs, int4 dims,
                          int4 perm, int to_layout) {
  const int dc[4] = {dims.x, dims.y, dims.z, dims.w};
  const int pm[4] = {perm.x, perm.y, perm.z, perm.w};
  long long n = 4;
  for (int k = 0; k < nlegs; ++k) n *= dc[k];
  // strides of the canonical legs inside the layout
  long long sl[4] = {0, 0, 0, 0};
  long long st = 4;
  for (int k = nlegs - 1; k >= 0; --k) { sl[pm[k]] = st; st *= dc[pm[k]]; }
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    long long rem = e >> 2, dst = e & 3;
    for (int k = nlegs - 1; k >= 0; --k) {
      long long j = rem % dc[k];
      rem /= dc[k];
      dst += j * sl[k];
    }
    if (to_layout) out[dst] = in[e];
    else out[e] = in[dst];
  }
}

template <typename T>
cudaError_t launch_permute(const void* in, void* out, int nlegs, const int* dims_canon, const int* perm,
                           int to_layout, cudaStream_t s) {
  int4 d = make_int4(nlegs > 0 ? dims_canon[0] : 1, nlegs > 1 ? dims_canon[1] : 1,
                     nlegs > 2 ? dims_canon[2] : 1, nlegs > 3 ? dims_canon[3] : 1);
  int4 p = make_int4(nlegs > 0 ? perm[0] : 0, nlegs > 1 ? perm[1] : 0, nlegs > 2 ? perm[2] : 0,
                     nlegs > 3 ? perm[3] : 0);
  k_permute<T><<<1024, 256, 0, s>>>(static_cast<const T*>(in), static_cast<T*>(out), nlegs, d, p,
                                    to_layout);
  return cudaGetLastError();
}

template cudaError_t launch_leg_contract<float>(const LegItem*, int, int, void* const*,
                                                const int*, cudaStream_t);
template cudaError_t launch_leg_contract<double>(const LegItem*, int, int, void* const*,
                                                 const int*, cudaStream_t);
template cudaError_t launch_gram_leg<float>(const GramLegItem*, int, int, int, void* const*,
                                            const int*, cudaStream_t);
template cudaError_t launch_gram_leg<double>(const GramLegItem*, int, int, int, void* const*,
                                             const int*, cudaStream_t);
template cudaError_t launch_permute<float>(const void*, void*, int, const int*, const int*, int,
                                           cudaStream_t);
template cudaError_t launch_permute<double>(const void*, void*, int, const int*, const int*, int,
                                            cudaStream_t);

}  // namespace pepo
