// Fifth-generation tensor-core (tcgen05) contractions for the FP32-storage
// mixed-precision mode: the leg contraction and the free-leg Gram of the BP
// message products (Eq. 13) and of the absorb step (Sec. 2.5 step 1).
//
//   k_leg_umma   out[o, i, q] = sum_j A[i, j] in[o, j, q]
//   k_gram_umma  S[i, i'] = sum_k (Xh[i,k] Xh[i',k] + 2 Xh[i,k] Xl[i',k])
//                over one K-range (split) of k = (o, q); the reduction sums the
//                splits and symmetrises: G = (S + S^T) / 2 = sum w^2 X X^T up
//                to the dropped lo*lo term.
//
// Split precision (three-product TF32): every FP32 operand x is split as
// x = hi + lo with hi = tf32(x) (round to nearest) and lo = x - hi (exact in
// FP32; the tensor core keeps its leading 11 bits).  A product a*b is taken as
// ah*bh + ah*bl + al*bh; the dropped al*bl and the truncation of lo are
// ~2^-21 relative.  For the leg contraction the hi and lo rows of the small
// matrix A are stacked along N, so one MMA of width 2N gives [ah*bh | ah*bl]
// and a second of width N adds al*bh to the first half.  For the Gram both
// operands are the same tile X, stacked as [Xh; Xl] along N: one MMA gives
// [Xh Xh^T | Xh Xl^T] and the symmetrisation supplies Xl Xh^T.
//
// Pipeline (one persistent CTA per SM; 512 threads, the Gram 768):
//   warp 0        allocates tensor memory; waits as a whole and elects the lane
//                 that issues a chunk's MMAs and the commits that release
//                 shared-memory stages and hand finished accumulators to the
//                 epilogue
//   warp 1        reconstruct: bulk copies of the packed W blocks
//   warps 4-7     epilogue: tcgen05.ld of the accumulator (warp w reads TMEM
//                 lanes 32 (w % 4) .. +31), store to global memory (leg) or
//                 add into compensated FP32 sums in shared memory (Gram)
//   warps 8-      converters in groups of 128 threads that take turns with the
//                 chunks (leg, reconstruct: two groups, the next chunk of each
//                 in a second set of registers; Gram: up to four groups, one
//                 set each): coalesced global loads, split, and 16-byte
//                 conflict-free stores into the swizzled K-major layout the MMA
//                 descriptors describe (below)
// Stages and accumulators are handed over with mbarriers.  Every wait is
// bounded (a few seconds of %globaltimer); on expiry the kernel records bit 0
// in *err (bit 1 marks a reconstruct item without its packed-W workspace),
// every role leaves its loop, the MMA issuer drains its outstanding
// MMAs (bounded), tensor memory is freed and the kernel returns.
//
// Shared-memory operand layout: K-major with the 128-byte swizzle.  A row of
// an operand holds the 32 FP32 (TF32) values of one K chunk in 128 bytes;
// 8 rows form a 1024-byte atom (atoms SBO = 1024 bytes apart along M/N); the
// 16-byte piece c of row r sits at piece position c ^ (r % 8).  One MMA
// covers K = 8 (32 bytes): its descriptor starts 32 bytes further per K step
// inside the atom (the hardware applies the XOR to the absolute address, so
// every tile is 1024-byte aligned).  Element (n, k) of a tile sits at
// (n / 8) 1024 + (n % 8) 128 + (((k / 4) ^ (n % 8)) 16) + (k % 4) 4.
#include "kernels.h"

namespace pepo {
namespace um {

constexpr int kThreads = 512;
constexpr int kConv = 256;              // converter threads (warps 8..15)
constexpr int kGroup = 128;             // converter threads of one chunk: two groups take turns
// The Gram's groups of converters: four, one chunk in registers each, or as many as
// there are stages (a group may wait for a stage's next release only, so two
// groups never wait for the same stage).
constexpr int kGramGroups = 4;
constexpr int kGramThreads = 256 + kGramGroups * kGroup;
constexpr int kM = 128;                 // accumulator rows = TMEM lanes
constexpr int kKC = 32;                 // K values per staged chunk
constexpr int kTmemCols = 512;          // two accumulators of 256 columns
// Gram chunks per FP32 accumulator run (1024 K terms summed in TMEM before
// the compensated shared-memory sums take them): the FP32 rounding of a run
// is ~1e-6 of its sum in the worst case, below the split-TF32 product error,
// and the epilogue's pass over the accumulator is paid once per run
constexpr int kRun = 32;
constexpr unsigned long long kDrainNs = 2000000000ull;   // bound of the exit drains

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long gtimer() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait for the phase of parity `parity`; false once the CTA aborts.
// `limit` (ns of %globaltimer) is the launch's wait limit; on expiry the wait
// records bit 0 in *err and raises the CTA's abort flag.
__device__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, int* err,
                          unsigned long long limit) {
  if (mbar_try(b, parity)) return true;
  const unsigned long long t0 = gtimer();
  while (true) {
    if (mbar_try(b, parity)) return true;
    if (*abort_flag) return false;
    if (gtimer() - t0 > limit) {
      *abort_flag = 1;
      atomicOr(err, 1);
      return false;
    }
  }
}

// Wait on the way out, also after an abort: the CTA's own MMAs and bulk
// copies in flight complete before its tensor and shared memory are released.
// Bounded by kDrainNs (they finish within microseconds); bit 2 in *err if not.
__device__ void mbar_drain(uint64_t* b, uint32_t parity, int* err) {
  const unsigned long long t0 = gtimer();
  while (!mbar_try(b, parity)) {
    if (gtimer() - t0 > kDrainNs) {
      atomicOr(err, 4);
      return;
    }
  }
}

// warp-uniform wait (every lane agrees, so the warp leaves a loop together)
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, int* err,
                                          unsigned long long limit) {
  const bool ok = mbar_wait(b, parity, abort_flag, err, limit);
  return __all_sync(0xffffffffu, ok);
}
// one arrival per warp once every lane's shared-memory writes are ordered
// before it (the lanes' proxy fences precede the warp barrier)
__device__ __forceinline__ void warp_arrive(uint64_t* b) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(b);
}

__device__ __forceinline__ void mbar_arrive_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
// global -> shared bulk copy (16-byte aligned, size a multiple of 16) that
// completes `bytes` of the barrier's transaction count
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* b) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   su32(dst)),
               "l"(src), "r"(bytes), "r"(su32(b))
               : "memory");
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t* slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(slot)),
               "r"(kTmemCols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t taddr) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(kTmemCols) : "memory");
}

// shared-memory matrix descriptor: K-major, 128-byte swizzle, atoms 1024
// bytes apart (the leading offset is unused for this layout: one atom spans
// the MMA's K).  The high word is the same for every operand; the low word is
// the address in 16-byte units and the leading offset (16 bytes, unused), so
// a K step of 32 bytes adds 2 to it.
constexpr uint32_t kDescHi = (1024u >> 4)          // stride byte offset: 8-row atoms
                             | (1u << 14)          // descriptor version of the sm_100 family
                             | (2u << 29);         // layout: 128-byte swizzle
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFFu) | (1u << 16); }
// byte offset of the 16-byte piece `piece` (K / 4) of row `row` in a tile
__host__ __device__ __forceinline__ uint32_t swz(int row, int piece) {
  return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((piece ^ (row & 7)) << 4));
}
// instruction descriptor: kind::tf32, FP32 accumulator, A and B TF32 K-major
__device__ __forceinline__ uint32_t idesc_tf32(int m, int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
// D (+)= A B over one K step; a and b are descriptor low words
__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 da, {%1, %5};\n\t"
      "mov.b64 db, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], da, db, %3, p;\n\t}\n" ::"r"(d_tmem),
      "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(kDescHi)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(b))
               : "memory");
}
// One lane of the converged warp, always the same one.  The MMA warp runs its
// loops and waits as a whole and elects the issuing lane around each chunk's
// MMAs, so that descriptors and loop state stay warp-uniform: a branch on the
// lane around the whole role kept them per thread, and the issue of a chunk
// then took longer (1180 cycles for 8 MMAs) than the tensor core needs (510).
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok));
  return ok != 0;
}
// the three TF32 products of one K chunk of a split operand pair (KS K steps):
// [Dhh | Dhl] (+)= Ahi [Bhi; Blo]^T, Dhh += Alo Bhi^T
template <int KS>
__device__ __forceinline__ void mma_split(uint32_t d_tmem, uint32_t ah, uint32_t al, uint32_t b, uint32_t id_wide,
                                          uint32_t id_half, uint32_t acc0) {
#pragma unroll
  for (int st = 0; st < KS; ++st) {
    mma_tf32(d_tmem, ah + 2u * st, b + 2u * st, id_wide, st > 0 ? 1u : acc0);
    mma_tf32(d_tmem, al + 2u * st, b + 2u * st, id_half, 1u);
  }
}
__device__ __forceinline__ void mma_split_chunk(int ksteps, uint32_t d_tmem, uint32_t ah, uint32_t al, uint32_t b,
                                                uint32_t id_wide, uint32_t id_half, uint32_t acc0) {
  switch (ksteps) {
    case 4: mma_split<4>(d_tmem, ah, al, b, id_wide, id_half, acc0); break;
    case 3: mma_split<3>(d_tmem, ah, al, b, id_wide, id_half, acc0); break;
    case 2: mma_split<2>(d_tmem, ah, al, b, id_wide, id_half, acc0); break;
    default: mma_split<1>(d_tmem, ah, al, b, id_wide, id_half, acc0); break;
  }
}
// 32 TMEM lanes x 16 consecutive 32-bit columns; thread t receives lane
// (lane base + t).  The registers are valid after tmem_wait32.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// completes outstanding tcgen05.ld of two 16-column blocks at once; both
// register sets are threaded through so no use is scheduled before the wait
__device__ __forceinline__ void tmem_wait32(uint32_t* r, uint32_t* q) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), "+r"(q[6]),
                 "+r"(q[7]), "+r"(q[8]), "+r"(q[9]), "+r"(q[10]), "+r"(q[11]), "+r"(q[12]), "+r"(q[13]), "+r"(q[14]),
                 "+r"(q[15])
               :
               : "memory");
}
__device__ __forceinline__ float tf32_hi(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__host__ __device__ inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// ============================================================ leg contraction
struct LegPlan {
  const float* in;
  float* out;
  const double* A;
  unsigned R, Q;       // rows (o, q) of the item, values between two j
  int J, Jout, K8, N16, nkc, lda;
  int kb, kr;          // K steps of 8 a chunk: kb, one more in the first kr chunks
  // first K value of chunk kc.  The chunks are as even as their steps allow (J = 100: 32,
  // 24, 24, 24 and not 32, 32, 32, 8): the loads of a group's next chunk hide
  // behind the conversion of this one, and a chunk of 8 hides nothing.
  __device__ __forceinline__ int k0(int kc) const { return 8 * (kb * kc + min(kc, kr)); }
  __device__ __forceinline__ int steps(int kc) const { return kb + (kc < kr ? 1 : 0); }
};

__device__ inline unsigned leg_rows(const LegItem& it, const int* ival, unsigned& Q, int& J) {
  unsigned O = 1;
  Q = 4;
  J = 1;
#pragma unroll
  for (int k = 0; k < PEPO_MAXLEG; ++k) {
    const int dk = (k < it.in.nlegs) ? ival[it.in.dim[k]] : 1;
    if (k == it.leg) J = dk;
    else if (k < it.leg) O *= dk;
    else Q *= dk;
  }
  return O * Q;
}
__device__ __noinline__ void leg_plan(const LegItem* items, int i, void* const* ptrs, const int* ival, LegPlan& L) {
  const LegItem& it = items[i];
  L.R = leg_rows(it, ival, L.Q, L.J);
  L.Jout = ival[it.out_dim];
  L.K8 = round_up(L.J, 8);
  // N >= 16: a factor of rank 0 (a message that is not finite) still issues MMAs
  L.N16 = round_up(L.Jout > 0 ? L.Jout : 1, 16);
  L.nkc = (L.K8 + kKC - 1) / kKC;
  L.kb = L.nkc > 0 ? L.K8 / 8 / L.nkc : 0;
  L.kr = L.K8 / 8 - L.kb * L.nkc;
  L.in = static_cast<const float*>(ptrs[it.in.ref]);
  L.out = static_cast<float*>(ptrs[it.out_ref]);
  L.A = it.A;
  L.lda = it.lda;
}

// The CTA's tiles of the launch, item by item: lo, lo + step, .. (cnt of them) of
// `item`.  Tile g of the launch goes to CTA g mod grid where the items are large
// (at least 8 tiles per CTA on average): the CTAs then work on neighbouring
// tiles, whose 512-byte pieces of a row share DRAM pages, instead of streaming
// through 152 places of the tensor at once.  Small items are cut into
// contiguous ranges, so that a CTA sees few of them (each brings its own small
// matrix).
struct ItemRange {
  int item;
  unsigned lo, cnt, step, t, t1;
  __device__ void start(const unsigned* toff, int n) {
    const unsigned long long T = toff[n];
    item = -1;
    if (T >= 8ull * n * gridDim.x) {
      step = gridDim.x;
      t = blockIdx.x;
      t1 = (unsigned)T;
    } else {
      step = 1;
      t = (unsigned)(T * blockIdx.x / gridDim.x);
      t1 = (unsigned)(T * (blockIdx.x + 1) / gridDim.x);
    }
  }
  __device__ bool next(const unsigned* toff, int n) {      // false when the CTA is done
    if (t >= t1) return false;
    if (item < 0) item = 0;
    while (item + 1 < n && toff[item + 1] <= t) ++item;
    lo = t - toff[item];
    cnt = (min(t1, toff[item + 1]) - t + step - 1) / step;
    t += cnt * step;
    return true;
  }
};

// Shared-memory plan of k_leg_umma for a given chi bound.
struct LegSmem {
  int k8max, n16max, stages;
  size_t b_bytes, stage_bytes, bar_off, total;
};
__host__ __device__ inline LegSmem leg_smem(int chimax) {
  LegSmem p;
  p.k8max = round_up(chimax, 8);
  p.n16max = round_up(chimax, 16);
  // [Ah; Al] of the small matrix: one (2 N16 rows x 128 B) block per K chunk
  p.b_bytes = (size_t)((p.k8max + kKC - 1) / kKC) * (2 * p.n16max) * 128;
  p.stage_bytes = 2 * (size_t)kM * 128;                             // hi + lo tile, 2 x 16 KB
  const size_t budget = 227 * 1024 - 1024 - 8 * kMaxItems - 512;
  p.stages = (int)((budget - p.b_bytes) / p.stage_bytes);
  if (p.stages > 4) p.stages = 4;
  p.bar_off = p.b_bytes + p.stages * p.stage_bytes;
  p.total = p.bar_off + 512 + 8 * (size_t)(kMaxItems + 1) + 1024;   // + alignment slack
  return p;
}

struct LegBars {
  uint64_t full[4], empty[4], accfull[2], accempty[2], bfull, bfree, drain;
  uint32_t tmem;
  int abort_flag;
};

__global__ void __launch_bounds__(kThreads, 1)
k_leg_umma(const LegItem* __restrict__ items, int n_items, int chimax, void* const* ptrs,
           const int* __restrict__ ival, int* err, unsigned long long lim) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const LegSmem P = leg_smem(chimax);
  unsigned char* Bs = smem;                          // [Ah; Al] small matrix
  unsigned char* As = smem + P.b_bytes;              // stages: hi tile, lo tile
  LegBars* bars = reinterpret_cast<LegBars*>(smem + P.bar_off);
  unsigned* toff = reinterpret_cast<unsigned*>(smem + P.bar_off + 512);
  volatile int* abort_flag = &bars->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NS = P.stages;

  for (int i = tid; i < n_items; i += kThreads) {
    unsigned Q;
    int J;
    toff[i + 1] = (leg_rows(items[i], ival, Q, J) + kM - 1) / kM;
  }
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) { mbar_init(&bars->full[s], kGroup / 32); mbar_init(&bars->empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&bars->accfull[b], 1); mbar_init(&bars->accempty[b], 4); }
    mbar_init(&bars->bfull, kConv / 32);
    mbar_init(&bars->bfree, 1);
    mbar_init(&bars->drain, 1);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(&bars->tmem);
  tc_before();
  __syncthreads();
  if (tid == 0) {
    toff[0] = 0;
    for (int i = 0; i < n_items; ++i) toff[i + 1] += toff[i];
  }
  __syncthreads();
  tc_after();
  const uint32_t tmem = bars->tmem;
  ItemRange rg;
  rg.start(toff, n_items);
  LegPlan L;

  if (warp == 0) {
    // ------------------------------------------------------------ MMA issuer
    unsigned tc = 0;
    int st_i = 0;            // operand stage and its phase parity (advanced per chunk)
    uint32_t st_ph = 0;
    bool ok = true;
    for (unsigned item_n = 0; ok && rg.next(toff, n_items); ++item_n) {
      leg_plan(items, rg.item, ptrs, ival, L);
      const int N16 = L.N16, nkc = L.nkc;
      const uint32_t bstep = (uint32_t)(2 * N16) * 8;    // B block per K chunk (16-byte units)
      const uint32_t id_wide = idesc_tf32(kM, 2 * N16), id_half = idesc_tf32(kM, N16);
      if (!warp_wait(&bars->bfull, item_n & 1u, abort_flag, err, lim)) break;
      tc_after();
      for (unsigned i = 0; i < rg.cnt && ok; ++i, ++tc) {
        const int b = (int)(tc & 1);
        if (!warp_wait(&bars->accempty[b], ((tc >> 1) & 1u) ^ 1u, abort_flag, err, lim)) { ok = false; break; }
        tc_after();
        const uint32_t d_tmem = tmem + (uint32_t)(b * 256);
        uint32_t db = desc_lo(su32(Bs));
        for (int kc = 0; kc < nkc; ++kc, db += bstep) {
          const int s = st_i;
          if (!warp_wait(&bars->full[s], st_ph, abort_flag, err, lim)) { ok = false; break; }
          if (++st_i == NS) { st_i = 0; st_ph ^= 1u; }
          tc_after();
          const uint32_t da = desc_lo(su32(As) + (uint32_t)s * (uint32_t)P.stage_bytes);
          if (elect_one()) {
            mma_split_chunk(L.steps(kc), d_tmem, da, da + (uint32_t)(P.stage_bytes / 32), db, id_wide,
                            id_half, kc > 0 ? 1u : 0u);
            mma_commit(&bars->empty[s]);
          }
          __syncwarp();
        }
        if (ok && elect_one()) mma_commit(&bars->accfull[b]);
        __syncwarp();
      }
      if (ok && elect_one()) mma_commit(&bars->bfree);
      __syncwarp();
    }
    // every issued MMA completes before tensor memory is released
    if (elect_one()) {
      mma_commit(&bars->drain);
      mbar_drain(&bars->drain, 0, err);
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 8) {
    // -------------------------------------------------------------- epilogue
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    unsigned tc = 0;
    bool ok = true;
    while (ok && rg.next(toff, n_items)) {
      leg_plan(items, rg.item, ptrs, ival, L);
      const int N16 = L.N16, Jout = L.Jout;
      const unsigned Q = L.Q;
      for (unsigned i = 0, tile = rg.lo; i < rg.cnt; ++i, tile += rg.step, ++tc) {
        const int b = (int)(tc & 1);
        if (!warp_wait(&bars->accfull[b], (tc >> 1) & 1u, abort_flag, err, lim)) { ok = false; break; }
        tc_after();
        const unsigned r = tile * kM + row;
        const bool valid = r < L.R;
        const unsigned o = valid ? r / Q : 0u, q = valid ? r - o * Q : 0u;
        float* dst = L.out + (long long)o * Jout * Q + q;
        const uint32_t tbase = tmem + lane_base + (uint32_t)(b * 256);
        // 16-column blocks; the TMEM loads of block i+1 are in flight while
        // block i is stored (two register sets, unrolled so none is copied)
        uint32_t a1[16], a2[16], b1[16], b2[16];
        auto store_blk = [&](const uint32_t* p1, const uint32_t* p2, int c0) {
          if (!valid) return;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            if (c0 + i < Jout) *dst = __uint_as_float(p1[i]) + __uint_as_float(p2[i]);
            dst += Q;
          }
        };
        tmem_ld16(tbase, a1);
        tmem_ld16(tbase + (uint32_t)N16, a2);
        tmem_wait32(a1, a2);
        for (int c0 = 0; c0 < N16; c0 += 32) {
          const bool m1 = c0 + 16 < N16;
          if (m1) {
            tmem_ld16(tbase + (uint32_t)(c0 + 16), b1);
            tmem_ld16(tbase + (uint32_t)(N16 + c0 + 16), b2);
          }
          store_blk(a1, a2, c0);
          if (!m1) break;
          tmem_wait32(b1, b2);
          const bool m2 = c0 + 32 < N16;
          if (m2) {
            tmem_ld16(tbase + (uint32_t)(c0 + 32), a1);
            tmem_ld16(tbase + (uint32_t)(N16 + c0 + 32), a2);
          }
          store_blk(b1, b2, c0 + 16);
          if (!m2) break;
          tmem_wait32(a1, a2);
        }
        tc_before();
        warp_arrive(&bars->accempty[b]);
      }
    }
  } else if (warp >= 8) {
    // ------------------------------------------------------------ converters
    // This thread owns row r of every other chunk: 32 coalesced 4-byte loads
    // (the lanes of a warp read 32 consecutive rows), then 16-byte stores into
    // the K-major layout (8 consecutive rows per quarter warp: no bank conflicts).
    // The loads of the group's next chunk are in flight while one is converted.
    const int ct = tid - 256, grp = ct / kGroup, r = ct % kGroup;
    unsigned n = 0;                                   // chunks of the CTA before this item
    bool ok = true;
    for (unsigned item_n = 0; ok && rg.next(toff, n_items); ++item_n) {
      leg_plan(items, rg.item, ptrs, ival, L);
      const int nkc = L.nkc, J = L.J;
      const unsigned Q = L.Q;
      const unsigned total = rg.cnt * (unsigned)nkc;
      unsigned j = (n ^ (unsigned)grp) & 1u;           // this group's first chunk of the item
      unsigned nn = n + j;                             // its number in the CTA
      n += total;
      // load cursor: chunk (tile, kc) and this thread's source row
      unsigned tile = rg.lo, lj = j;
      int kc = (int)j;
      const float* src = L.in;
      bool valid = false;
      auto enter = [&]() {
        while (kc >= nkc) { kc -= nkc; tile += rg.step; }
        const unsigned rr = tile * kM + r;
        valid = rr < L.R;
        const unsigned o = valid ? rr / Q : 0u;
        src = L.in + (long long)o * J * Q + (valid ? rr - o * Q : 0u);
      };
      auto load = [&](float4 (&v)[8]) {
        const int k0 = L.k0(kc);
        const int m = valid ? min(J - k0, 8 * L.steps(kc)) : 0;   // values of this row in the chunk
        const float* p = src + (long long)k0 * Q;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (4 * u < m) v[u].x = __ldg(p);
          p += Q;
          if (4 * u + 1 < m) v[u].y = __ldg(p);
          p += Q;
          if (4 * u + 2 < m) v[u].z = __ldg(p);
          p += Q;
          if (4 * u + 3 < m) v[u].w = __ldg(p);
          p += Q;
        }
        lj += 2;
        kc += 2;
        if (lj < total) enter();
      };
      int ckc = (int)(j % (unsigned)nkc);              // K chunk of the chunk being converted
      auto convert = [&](const float4 (&v)[8]) -> bool {
        const unsigned s = nn % (unsigned)NS;
        if (!warp_wait(&bars->empty[s], ((nn / (unsigned)NS) & 1u) ^ 1u, abort_flag, err, lim)) return false;
        unsigned char* hi = As + (size_t)s * P.stage_bytes;
        unsigned char* lo = hi + P.stage_bytes / 2;
        const int kw = 8 * L.steps(ckc);               // columns the MMAs of this chunk read
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (4 * u < kw) {
            const uint32_t off = swz(r, u);
            const float4 x = v[u];
            const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
            *reinterpret_cast<float4*>(hi + off) = h;
            *reinterpret_cast<float4*>(lo + off) = make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
          }
        }
        fence_async_smem();
        warp_arrive(&bars->full[s]);
        nn += 2;
        ckc += 2;
        while (ckc >= nkc) ckc -= nkc;
        return true;
      };
      float4 v0[8], v1[8];
      if (j < total) {
        enter();
        load(v0);
      }
      // the item's small matrix [Ah; Al]: rows q < N16 hold hi(A[q, :]), rows N16 + q
      // hold lo(A[q, :]); one block of 2 N16 rows per 32-wide K chunk
      if (item_n > 0 && !warp_wait(&bars->bfree, (item_n - 1) & 1u, abort_flag, err, lim)) break;
      {
        const size_t bblk = (size_t)(2 * L.N16) * 128;
        const int K32 = nkc * kKC;
        for (int e = ct; e < L.N16 * K32; e += kConv) {
          const int q = e / K32, kk = e - q * K32;
          const int kc = kk / kKC, k = L.k0(kc) + kk % kKC;
          float x = 0.f;
          if (q < L.Jout && k < J && kk % kKC < 8 * L.steps(kc)) x = (float)L.A[(long long)q * L.lda + k];
          const float h = tf32_hi(x);
          unsigned char* blk = Bs + (size_t)kc * bblk + (size_t)(kk & 3) * 4;
          const int piece = (kk % kKC) >> 2;
          *reinterpret_cast<float*>(blk + swz(q, piece)) = h;
          *reinterpret_cast<float*>(blk + swz(q + L.N16, piece)) = x - h;
        }
        fence_async_smem();
        warp_arrive(&bars->bfull);
      }
      for (; j < total; j += 4) {
        if (j + 2 < total) load(v1);
        if (!convert(v0)) { ok = false; break; }
        if (j + 2 >= total) break;
        if (j + 4 < total) load(v0);
        if (!convert(v1)) { ok = false; break; }
      }
    }
  }
  tc_before();
  __syncthreads();
  if (warp == 0) {
    tc_after();
    tmem_free(tmem);
  }
}

// ============================================================ Gram (free leg)
// A free-leg Gram sums over the flattened (o, q): NQ quads of 4 values per row,
// Q4 per (o, row).  A chunk is 8 quads of every row; unit = (item, split) = a
// range of chunks.
struct GramUnit {
  const float* X;
  double* partial;
  long long FQ, Q;     // values between two o, between two rows
  unsigned Q4, NQ;
  int F, F8, s;
  unsigned c0, c1;     // chunks of the unit
};
__device__ inline void gram_extent(const GramLegItem& it, const int* ival, int& F, unsigned& O, unsigned& Q4) {
  F = 1;
  O = 1;
  Q4 = 1;
#pragma unroll
  for (int k = 0; k < PEPO_MAXLEG; ++k) {
    const int dk = (k < it.x.nlegs) ? ival[it.x.dim[k]] : 1;
    if (k == it.leg) F = dk;
    else if (k < it.leg) O *= dk;
    else Q4 *= dk;
  }
}
__device__ inline int gram_splits(unsigned O, unsigned Q4, int splits_max) {
  return gram_leg_splits_k((long long)O * Q4 * 4, splits_max, kGramLegRowsUmma);
}
// unit u through the prefix table of split counts
__device__ __noinline__ void gram_unit(GramUnit& g, long long u, const long long* uoff, int n, const GramLegItem* items,
                                       void* const* ptrs, const int* ival, int splits_max) {
  int i = 0;
  while (i + 1 < n && uoff[i + 1] <= u) ++i;
  const GramLegItem& it = items[i];
  unsigned O;
  gram_extent(it, ival, g.F, O, g.Q4);
  g.F8 = round_up(g.F, 8);
  g.Q = 4ll * g.Q4;
  g.FQ = g.Q * g.F;
  g.NQ = O * g.Q4;
  const unsigned long long NC = (g.NQ + 7) / 8, S = (unsigned long long)gram_splits(O, g.Q4, splits_max);
  g.s = (int)(u - uoff[i]);
  g.c0 = (unsigned)(NC * g.s / S);
  g.c1 = (unsigned)(NC * (g.s + 1) / S);
  g.X = static_cast<const float*>(ptrs[it.x.ref]);
  g.partial = it.partial;
}

struct GramSmem {
  int f8max, stages, ld;
  size_t stage_bytes, acc_off, bar_off, total;
};
__host__ __device__ inline GramSmem gram_smem(int chimax) {
  GramSmem p;
  p.f8max = round_up(chimax, 8);
  // [Xh; Xl] rows x 128 B; at least the 128 rows the A operand (M = 128) reads
  p.stage_bytes = (size_t)(2 * p.f8max > kM ? 2 * p.f8max : kM) * 128;
  p.ld = p.f8max + 1;                                               // odd row stride (words)
  const size_t acc_bytes = 2 * (size_t)p.f8max * p.ld * 4;          // sum + compensation
  const size_t budget = 227 * 1024 - 1024 - 8 * (kMaxItems + 1) - 512 - 1024;
  p.stages = acc_bytes < budget ? (int)((budget - acc_bytes) / p.stage_bytes) : 0;
  if (p.stages > 4) p.stages = 4;
  p.acc_off = p.stages * p.stage_bytes;
  p.bar_off = p.acc_off + acc_bytes;
  p.total = p.bar_off + 512 + 8 * (size_t)(kMaxItems + 1) + 1024 + 1024;
  return p;
}

struct GramBars {
  uint64_t full[4], empty[4], accfull[2], accempty[2], drain;
  uint32_t tmem;
  int abort_flag;
};

__global__ void __launch_bounds__(kGramThreads, 1)
k_gram_umma(const GramLegItem* __restrict__ items, int n_items, int splits_max, int chimax, void* const* ptrs,
            const int* __restrict__ ival, int* err, unsigned long long lim) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const GramSmem P = gram_smem(chimax);
  unsigned char* Xs = smem;
  float* acc = reinterpret_cast<float*>(smem + P.acc_off);
  float* cmp = acc + (size_t)P.f8max * P.ld;
  GramBars* bars = reinterpret_cast<GramBars*>(smem + P.bar_off);
  long long* uoff = reinterpret_cast<long long*>(smem + P.bar_off + 512);
  volatile int* abort_flag = &bars->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NS = P.stages;

  for (int i = tid; i < n_items; i += kGramThreads) {
    int F;
    unsigned O, Q4;
    gram_extent(items[i], ival, F, O, Q4);
    uoff[i + 1] = gram_splits(O, Q4, splits_max);
  }
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) { mbar_init(&bars->full[s], kGroup / 32); mbar_init(&bars->empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&bars->accfull[b], 1); mbar_init(&bars->accempty[b], 4); }
    mbar_init(&bars->drain, 1);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  // zero the operand stages once: rows [F, F8) stay zero-filled by the
  // converters, everything else is rewritten before use
  for (size_t e = tid; e < (size_t)NS * P.stage_bytes / 16; e += kGramThreads)
    reinterpret_cast<float4*>(Xs)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (warp == 0) tmem_alloc(&bars->tmem);
  tc_before();
  __syncthreads();
  if (tid == 0) {
    uoff[0] = 0;
    for (int i = 0; i < n_items; ++i) uoff[i + 1] += uoff[i];
  }
  __syncthreads();
  tc_after();
  const uint32_t tmem = bars->tmem;
  const long long U = uoff[n_items];

  if (warp == 0) {
    // ------------------------------------------------------------ MMA issuer
    GramUnit g;
    long long rc = 0;
    int st_i = 0;            // operand stage and its phase parity (advanced per chunk)
    uint32_t st_ph = 0;
    bool ok = true;
    for (long long u = blockIdx.x; u < U && ok; u += gridDim.x) {
      gram_unit(g, u, uoff, n_items, items, ptrs, ival, splits_max);
      const uint32_t id = idesc_tf32(kM, 2 * g.F8);
      for (unsigned c = g.c0; c < g.c1 && ok;) {
        const int b = (int)(rc & 1);
        if (!warp_wait(&bars->accempty[b], (uint32_t)(((rc >> 1) & 1) ^ 1), abort_flag, err, lim)) { ok = false; break; }
        tc_after();
        const uint32_t d_tmem = tmem + (uint32_t)(b * 256);
        const unsigned cend = min(g.c1, c + kRun);
        for (unsigned cr = c; cr < cend; ++cr) {
          const int s = st_i;
          if (!warp_wait(&bars->full[s], st_ph, abort_flag, err, lim)) { ok = false; break; }
          if (++st_i == NS) { st_i = 0; st_ph ^= 1u; }
          tc_after();
          const uint32_t dx = desc_lo(su32(Xs) + (uint32_t)s * (uint32_t)P.stage_bytes);
          if (elect_one()) {
            const uint32_t acc0 = cr > c ? 1u : 0u;
#pragma unroll
            for (uint32_t st = 0; st < kKC / 8; ++st)
              mma_tf32(d_tmem, dx + 2u * st, dx + 2u * st, id, st > 0 ? 1u : acc0);
            mma_commit(&bars->empty[s]);
            if (cr + 1 == cend) mma_commit(&bars->accfull[b]);
          }
          __syncwarp();
        }
        ++rc;
        c = cend;
      }
    }
    if (elect_one()) {
      mma_commit(&bars->drain);
      mbar_drain(&bars->drain, 0, err);
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 8) {
    // -------------------------------------------------------------- epilogue
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    GramUnit g;
    long long rc = 0;
    bool ok = true;
    for (long long u = blockIdx.x; u < U && ok; u += gridDim.x) {
      gram_unit(g, u, uoff, n_items, items, ptrs, ival, splits_max);
      const int F = g.F, F8 = g.F8;
      const bool live_row = row < F;
      if (live_row)
        for (int c0 = 0; c0 < F8; ++c0) { acc[(size_t)row * P.ld + c0] = 0.f; cmp[(size_t)row * P.ld + c0] = 0.f; }
      for (unsigned c = g.c0; c < g.c1; c += kRun) {
        const int b = (int)(rc & 1);
        if (!warp_wait(&bars->accfull[b], (uint32_t)((rc >> 1) & 1), abort_flag, err, lim)) { ok = false; break; }
        tc_after();
        const uint32_t tbase = tmem + lane_base + (uint32_t)(b * 256);
        for (int c0 = 0; c0 < F8; c0 += 16) {
          uint32_t v1[16], v2[16];
          tmem_ld16(tbase + (uint32_t)c0, v1);
          tmem_ld16(tbase + (uint32_t)(F8 + c0), v2);
          tmem_wait32(v1, v2);
          if (live_row) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int col = c0 + i;
              if (col < F) {
                // compensated (Kahan) FP32 sum of S += Xh Xh^T + 2 Xh Xl^T
                float* pa = acc + (size_t)row * P.ld + col;
                float* pc = cmp + (size_t)row * P.ld + col;
                const float y = (__uint_as_float(v1[i]) + 2.f * __uint_as_float(v2[i])) - *pc;
                const float t = *pa + y;
                *pc = (t - *pa) - y;
                *pa = t;
              }
            }
          }
        }
        tc_before();
        warp_arrive(&bars->accempty[b]);
        ++rc;
      }
      if (!ok) break;
      if (live_row) {
        double* P0 = g.partial + (size_t)g.s * F * F + (size_t)row * F;
        for (int col = 0; col < F; ++col)
          P0[col] = (double)acc[(size_t)row * P.ld + col] - (double)cmp[(size_t)row * P.ld + col];
      }
    }
  } else if (warp >= 8) {
    // ------------------------------------------------------------ converters
    // This thread copies quad kq of the rows r0 + 16 u of every fourth chunk of
    // the unit: the eight lanes of a row read 128 consecutive bytes (or eight
    // consecutive o), store one swizzled 128-byte row without bank conflicts.
    // Bound: the latency of these loads.  A group requests its next chunk as soon
    // as the one before is stored, so three or four chunks are on their way.
    const int ct = tid - 256, grp = ct / kGroup, t = ct % kGroup;
    const int kq = t & 7, r0 = t >> 3;
    constexpr int MU = kM / (kGroup / 8);             // row steps of 16
    const unsigned G = (unsigned)min(kGramGroups, NS);
    unsigned n = 0;                                   // chunks of the CTA before this unit
    GramUnit g;
    bool ok = (unsigned)grp < G;
    for (long long u = blockIdx.x; u < U && ok; u += gridDim.x) {
      gram_unit(g, u, uoff, n_items, items, ptrs, ival, splits_max);
      unsigned c = g.c0 + ((unsigned)grp + G - n % G) % G;   // this group's first chunk
      unsigned nn = n + (c - g.c0);                    // its number in the CTA
      n += g.c1 - g.c0;
      unsigned qi = 8 * c + kq;
      const unsigned o = qi / g.Q4;
      unsigned q4 = qi - o * g.Q4;
      const float* src = g.X + (long long)o * g.FQ + 4ll * q4 + (long long)r0 * g.Q;
      // the same quad of the group's next chunk: dO o's and dq quads further on
      const unsigned dO = 8 * G / g.Q4, dq = 8 * G - dO * g.Q4;
      const long long step = (long long)dO * g.FQ + 4ll * dq, wrap = g.FQ - g.Q, rows16 = 16 * g.Q;
      const unsigned Q4 = g.Q4, NQ = g.NQ, c1 = g.c1;
      const int F = g.F, F8 = g.F8;
      auto load = [&](float4 (&v)[MU]) {
        const bool live = qi < NQ;
        const float* p = src;
#pragma unroll
        for (int i = 0; i < MU; ++i) {
          v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (live && r0 + 16 * i < F) v[i] = __ldg(reinterpret_cast<const float4*>(p));
          p += rows16;
        }
        qi += 8 * G;
        q4 += dq;
        src += step;
        if (q4 >= Q4) { q4 -= Q4; src += wrap; }
      };
      auto convert = [&](const float4 (&v)[MU]) -> bool {
        const unsigned s = nn % (unsigned)NS;
        if (!warp_wait(&bars->empty[s], ((nn / (unsigned)NS) & 1u) ^ 1u, abort_flag, err, lim)) return false;
        unsigned char* st = Xs + (size_t)s * P.stage_bytes;
#pragma unroll
        for (int i = 0; i < MU; ++i) {
          const int r = r0 + 16 * i;
          if (r < F8) {
            const float4 x = v[i];
            const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
            *reinterpret_cast<float4*>(st + swz(r, kq)) = h;
            *reinterpret_cast<float4*>(st + swz(r + F8, kq)) = make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
          }
        }
        fence_async_smem();
        warp_arrive(&bars->full[s]);
        nn += G;
        return true;
      };
      float4 v[MU];
      if (c < c1) load(v);
      for (; c < c1; c += G) {
        if (!convert(v)) { ok = false; break; }
        if (c + G < c1) load(v);
      }
    }
  }
  tc_before();
  __syncthreads();
  if (warp == 0) {
    tc_after();
    tmem_free(tmem);
  }
}

// ================================================================ reconstruct
// out[perm(r), c] = sum_k in[r, k] W[k, c]: rows r = environment index of the
// site tensor (cut leg last), k = (cut, Pauli), c = (new cut, Pauli) written
// into the next update's layout.  Tiles are (128 rows, one N block of at most
// 128 columns); both operands stream in 32-wide K chunks: A through the
// converters (row-contiguous, 16-byte loads), B = [hi(W^T); lo(W^T)] of the
// tile's N block as one bulk copy of a block pre-packed by k_pack_w (the
// swizzled shared-memory image, so the copy is linear).
struct RecPlan {
  const float* in;
  float* out;
  const double* W;
  const float* Wp;
  unsigned R, nrb;         // rows, row blocks of 128
  int n, np, K8, nkc, nnb, NB, ldw;
  // Row r of the launch is (a0, a1, a2), a2 fastest, over the (up to three) row legs
  // ordered so that the one that is innermost in the output is a2: the lanes of
  // a warp then write 16-byte neighbours.
  unsigned d1, d2;                 // extents of a1, a2
  unsigned rs0, rs1, rs2;          // their strides among the input's rows
  long long os0, os1, os2, ocut;   // and in the output; the new cut leg's
};

__device__ inline unsigned rec_rows(const ReconItem& it, const int* ival) {
  unsigned R = 1;
#pragma unroll
  for (int i = 0; i < PEPO_MAXLEG; ++i)
    if (i + 1 < it.in.nlegs) R *= (unsigned)ival[it.in.dim[i]];
  return R;
}
__device__ inline void rec_blocks(int np, int& nnb, int& NB) {
  nnb = (np + 127) / 128;
  NB = round_up((np + nnb - 1) / nnb, 8);
}
__device__ __noinline__ void rec_plan(const ReconItem* items, int i, void* const* ptrs, const int* ival, RecPlan& D) {
  const ReconItem& it = items[i];
  const int nl = it.in.nlegs, cut = nl - 1;
  const int chin = ival[it.new_dim];
  D.n = 4 * ival[it.in.dim[cut]];
  D.np = 4 * chin;
  D.R = rec_rows(it, ival);
  D.nrb = (D.R + kM - 1) / kM;
  D.K8 = round_up(D.n, 8);
  D.nkc = (D.K8 + kKC - 1) / kKC;
  rec_blocks(D.np, D.nnb, D.NB);
  // output stride of input leg l: 4 x the product of the output extents of the
  // legs that follow it in the output order out_perm
  long long os[PEPO_MAXLEG] = {0, 0, 0, 0};
  int dd[PEPO_MAXLEG] = {1, 1, 1, 1};
  long long st = 4;
  for (int kk = nl - 1; kk >= 0; --kk) {
    const int l = it.out_perm[kk];
    const int e = l == cut ? chin : ival[it.in.dim[l]];
    os[l] = st;
    dd[l] = e;
    st *= e;
  }
  D.ocut = os[cut];
  // the row legs, right-aligned in three places (missing ones: extent 1), the
  // output's innermost one moved to the end
  unsigned rs[PEPO_MAXLEG] = {0, 0, 0, 0};
  unsigned q = 1;
  for (int l = cut - 1; l >= 0; --l) { rs[l] = q; q *= (unsigned)dd[l]; }
  int leg[3] = {-1, -1, -1};
  const int inner = it.out_perm[nl - 1];
  int at = 2;
  if (inner != cut && cut > 0) leg[at--] = inner;
  for (int l = cut - 1; l >= 0 && at >= 0; --l)
    if (l != inner) leg[at--] = l;
  D.rs0 = leg[0] >= 0 ? rs[leg[0]] : 0;
  D.os0 = leg[0] >= 0 ? os[leg[0]] : 0;
  D.rs1 = leg[1] >= 0 ? rs[leg[1]] : 0;
  D.os1 = leg[1] >= 0 ? os[leg[1]] : 0;
  D.d1 = leg[1] >= 0 ? dd[leg[1]] : 1;
  D.rs2 = leg[2] >= 0 ? rs[leg[2]] : 0;
  D.os2 = leg[2] >= 0 ? os[leg[2]] : 0;
  D.d2 = leg[2] >= 0 ? dd[leg[2]] : 1;
  D.in = static_cast<const float*>(ptrs[it.in.ref]);
  D.out = static_cast<float*>(ptrs[it.out_ref]);
  D.W = it.W;
  D.ldw = it.ldw;
  D.Wp = it.Wp;
}

struct RecSmem {
  int stages;
  size_t a_bytes, stage_bytes, bar_off, total;
};
__host__ __device__ inline RecSmem rec_smem() {
  RecSmem p;
  p.a_bytes = (size_t)kM * 128;                                   // 16 KB per hi / lo
  p.stage_bytes = 2 * p.a_bytes + (size_t)256 * 128;               // + [Bh; Bl], 2 NB <= 256 rows
  p.stages = 3;
  p.bar_off = p.stages * p.stage_bytes;
  p.total = p.bar_off + 512 + 8 * (size_t)(kMaxItems + 1) + 1024;
  return p;
}

struct RecBars {
  // full: the converter warps' A stages; wfull: the bulk copy of the W block
  // of the same stage (its own barrier, so that a CTA leaving early can wait
  // for exactly its copies in flight)
  uint64_t full[4], wfull[4], empty[4], accfull[2], accempty[2], drain;
  uint32_t tmem;
  int abort_flag;
};

__global__ void __launch_bounds__(kThreads, 1)
k_recon_umma(const ReconItem* __restrict__ items, int n_items, void* const* ptrs, const int* __restrict__ ival,
             int* err, unsigned long long lim) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const RecSmem P = rec_smem();
  RecBars* bars = reinterpret_cast<RecBars*>(smem + P.bar_off);
  unsigned* toff = reinterpret_cast<unsigned*>(smem + P.bar_off + 512);
  volatile int* abort_flag = &bars->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NS = P.stages;
  for (int i = tid; i < n_items; i += kThreads) {
    int nnb, NB;
    rec_blocks(4 * ival[items[i].new_dim], nnb, NB);
    toff[i + 1] = (rec_rows(items[i], ival) + kM - 1) / kM * nnb;
  }
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&bars->full[s], kGroup / 32);
      mbar_init(&bars->wfull[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(&bars->accfull[b], 1); mbar_init(&bars->accempty[b], 4); }
    mbar_init(&bars->drain, 1);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(&bars->tmem);
  tc_before();
  __syncthreads();
  if (tid == 0) {
    toff[0] = 0;
    for (int i = 0; i < n_items; ++i) toff[i + 1] += toff[i];
  }
  __syncthreads();
  tc_after();
  const uint32_t tmem = bars->tmem;
  ItemRange rg;
  rg.start(toff, n_items);
  RecPlan D;

  if (warp == 0) {
    // ------------------------------------------------------------ MMA issuer
    unsigned tc = 0;
    int st_i = 0;            // operand stage and its phase parity (advanced per chunk)
    uint32_t st_ph = 0;
    bool ok = true;
    while (ok && rg.next(toff, n_items)) {
      rec_plan(items, rg.item, ptrs, ival, D);
      const int NB = D.NB, K8 = D.K8, nkc = D.nkc;
      const uint32_t id_wide = idesc_tf32(kM, 2 * NB), id_half = idesc_tf32(kM, NB);
      for (unsigned i = 0; i < rg.cnt && ok; ++i, ++tc) {
        const int b = (int)(tc & 1);
        if (!warp_wait(&bars->accempty[b], ((tc >> 1) & 1u) ^ 1u, abort_flag, err, lim)) { ok = false; break; }
        tc_after();
        const uint32_t d_tmem = tmem + (uint32_t)(b * 256);
        for (int kc = 0; kc < nkc; ++kc) {
          const int s = st_i;
          if (!warp_wait(&bars->full[s], st_ph, abort_flag, err, lim)) { ok = false; break; }
          if (!warp_wait(&bars->wfull[s], st_ph, abort_flag, err, lim)) { ok = false; break; }
          if (++st_i == NS) { st_i = 0; st_ph ^= 1u; }
          tc_after();
          const uint32_t da = desc_lo(su32(smem) + (uint32_t)s * (uint32_t)P.stage_bytes);
          const uint32_t ab = (uint32_t)(P.a_bytes / 16);
          if (elect_one()) {
            mma_split_chunk(min(kKC, K8 - kc * kKC) / 8, d_tmem, da, da + ab, da + 2u * ab, id_wide, id_half,
                            kc > 0 ? 1u : 0u);
            mma_commit(&bars->empty[s]);
          }
          __syncwarp();
        }
        if (ok && elect_one()) mma_commit(&bars->accfull[b]);
        __syncwarp();
      }
    }
    if (elect_one()) {
      mma_commit(&bars->drain);
      mbar_drain(&bars->drain, 0, err);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------- W blocks, bulk copies
    if (lane == 0) {
      unsigned n = 0;          // copies issued
      bool ok = true;
      while (ok && rg.next(toff, n_items)) {
        rec_plan(items, rg.item, ptrs, ival, D);
        const uint32_t bytes = (uint32_t)(2 * D.NB) * 128u;
        for (unsigned i = 0, tile = rg.lo; i < rg.cnt && ok; ++i, tile += rg.step) {
          const float* blk = D.Wp + (size_t)(tile % (unsigned)D.nnb) * D.nkc * (size_t)(2 * D.NB) * 32;
          for (int kc = 0; kc < D.nkc; ++kc) {
            const unsigned s = n % (unsigned)NS;
            if (!mbar_wait(&bars->empty[s], ((n / (unsigned)NS) & 1u) ^ 1u, abort_flag, err, lim)) { ok = false; break; }
            if (D.Wp) {
              mbar_arrive_tx(&bars->wfull[s], bytes);
              bulk_g2s(smem + (size_t)s * P.stage_bytes + 2 * P.a_bytes, blk + (size_t)kc * (2 * D.NB) * 32, bytes,
                       &bars->wfull[s]);
            } else {   // no packed W workspace: flag it and keep the pipeline moving
              atomicOr(err, 2);
              mbar_arrive(&bars->wfull[s]);
            }
            ++n;
          }
        }
      }
      // no bulk copy may land after the kernel's shared memory is gone: the last
      // copy of every stage (a stage is armed again only after the MMAs that
      // consumed its previous copy)
      for (unsigned k = n > (unsigned)NS ? n - NS : 0; k < n; ++k)
        mbar_drain(&bars->wfull[k % (unsigned)NS], (k / (unsigned)NS) & 1u, err);
    }
    __syncwarp();
  } else if (warp >= 4 && warp < 8) {
    // -------------------------------------------------------------- epilogue
    const int row = 32 * (warp & 3) + lane;
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    unsigned tc = 0;
    bool ok = true;
    while (ok && rg.next(toff, n_items)) {
      rec_plan(items, rg.item, ptrs, ival, D);
      const int NB = D.NB;
      const long long ocut = D.ocut;
      for (unsigned i = 0, tile = rg.lo; i < rg.cnt; ++i, tile += rg.step, ++tc) {
        const int b = (int)(tc & 1);
        if (!warp_wait(&bars->accfull[b], (tc >> 1) & 1u, abort_flag, err, lim)) { ok = false; break; }
        tc_after();
        const unsigned rb = tile / (unsigned)D.nnb;
        const int nb = (int)(tile - rb * D.nnb);
        const unsigned r = rb * kM + row;
        const bool valid = r < D.R;
        const unsigned r1 = r / D.d2, i2 = r - r1 * D.d2, i0 = r1 / D.d1, i1 = r1 - i0 * D.d1;
        // first column of the tile (a multiple of 8): its cut index and Paulis
        float* dst = D.out + (i0 * D.os0 + i1 * D.os1 + i2 * D.os2) + (long long)(nb * NB / 4) * ocut;
        const int cols = valid ? min(NB, D.np - nb * NB) : 0;
        const uint32_t tbase = tmem + lane_base + (uint32_t)(b * 256);
        // 16-column blocks, loads of block i+1 in flight while block i is stored;
        // the four Paulis of a cut index are one 16-byte store
        uint32_t a1[16], a2[16], b1[16], b2[16];
        auto store_blk = [&](const uint32_t* p1, const uint32_t* p2, int c0) {
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            if (c0 + i < cols)
              *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(p1[i]) + __uint_as_float(p2[i]),
                                                            __uint_as_float(p1[i + 1]) + __uint_as_float(p2[i + 1]),
                                                            __uint_as_float(p1[i + 2]) + __uint_as_float(p2[i + 2]),
                                                            __uint_as_float(p1[i + 3]) + __uint_as_float(p2[i + 3]));
            dst += ocut;
          }
        };
        tmem_ld16(tbase, a1);
        tmem_ld16(tbase + (uint32_t)NB, a2);
        tmem_wait32(a1, a2);
        for (int c0 = 0; c0 < NB; c0 += 32) {
          const bool m1 = c0 + 16 < NB;
          if (m1) {
            tmem_ld16(tbase + (uint32_t)(c0 + 16), b1);
            tmem_ld16(tbase + (uint32_t)(NB + c0 + 16), b2);
          }
          store_blk(a1, a2, c0);
          if (!m1) break;
          tmem_wait32(b1, b2);
          const bool m2 = c0 + 32 < NB;
          if (m2) {
            tmem_ld16(tbase + (uint32_t)(c0 + 32), a1);
            tmem_ld16(tbase + (uint32_t)(NB + c0 + 32), a2);
          }
          store_blk(b1, b2, c0 + 16);
          if (!m2) break;
          tmem_wait32(a1, a2);
        }
        tc_before();
        warp_arrive(&bars->accempty[b]);
      }
    }
  } else if (warp >= 8) {
    // ------------------------------------------------------------ converters
    // This thread copies quad kq of the rows r0 + 16 u of every other chunk: the
    // eight lanes of a row read its 128 bytes and store one swizzled row.
    const int ct = tid - 256, grp = ct / kGroup, t = ct % kGroup;
    const int kq = t & 7, r0 = t >> 3;
    constexpr int MU = kM / (kGroup / 8);
    unsigned n = 0;                                   // chunks of the CTA before this item
    bool ok = true;
    while (ok && rg.next(toff, n_items)) {
      rec_plan(items, rg.item, ptrs, ival, D);
      const int nkc = D.nkc, K = D.n;
      const unsigned R = D.R;
      const unsigned total = rg.cnt * (unsigned)nkc;
      unsigned j = (n ^ (unsigned)grp) & 1u;
      unsigned nn = n + j;
      n += total;
      unsigned tile = rg.lo, lj = j;
      int kc = (int)j;
      const float* src[MU];                            // this thread's rows in the load cursor's tile (null: none)
      unsigned blk = ~0u;                              // row block they belong to
      auto enter = [&]() {
        while (kc >= nkc) { kc -= nkc; tile += rg.step; }
        const unsigned rb = tile / (unsigned)D.nnb;
        if (rb == blk) return;
        blk = rb;
#pragma unroll
        for (int i = 0; i < MU; ++i) {
          const unsigned r = rb * kM + r0 + 16 * i;
          const unsigned q = r / D.d2, a2 = r - q * D.d2, a0 = q / D.d1, a1 = q - a0 * D.d1;
          src[i] = r < R ? D.in + (long long)(a0 * D.rs0 + a1 * D.rs1 + a2 * D.rs2) * K + 4 * kq : nullptr;
        }
      };
      auto load = [&](float4 (&v)[MU]) {
        const int k = kc * kKC;
        const bool live = k + 4 * kq < K;
#pragma unroll
        for (int i = 0; i < MU; ++i) {
          v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (live && src[i]) v[i] = __ldg(reinterpret_cast<const float4*>(src[i] + k));
        }
        lj += 2;
        kc += 2;
        if (lj < total) enter();
      };
      auto convert = [&](const float4 (&v)[MU]) -> bool {
        const unsigned s = nn % (unsigned)NS;
        if (!warp_wait(&bars->empty[s], ((nn / (unsigned)NS) & 1u) ^ 1u, abort_flag, err, lim)) return false;
        unsigned char* hi = smem + (size_t)s * P.stage_bytes;
        unsigned char* lo = hi + P.a_bytes;
#pragma unroll
        for (int i = 0; i < MU; ++i) {
          const uint32_t off = swz(r0 + 16 * i, kq);
          const float4 x = v[i];
          const float4 h = make_float4(tf32_hi(x.x), tf32_hi(x.y), tf32_hi(x.z), tf32_hi(x.w));
          *reinterpret_cast<float4*>(hi + off) = h;
          *reinterpret_cast<float4*>(lo + off) = make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w);
        }
        fence_async_smem();
        warp_arrive(&bars->full[s]);
        nn += 2;
        return true;
      };
      float4 v0[MU], v1[MU];
      if (j < total) {
        enter();
        load(v0);
      }
      for (; j < total; j += 4) {
        if (j + 2 < total) load(v1);
        if (!convert(v0)) { ok = false; break; }
        if (j + 2 >= total) break;
        if (j + 4 < total) load(v0);
        if (!convert(v1)) { ok = false; break; }
      }
    }
  }
  tc_before();
  __syncthreads();
  if (warp == 0) {
    tc_after();
    tmem_free(tmem);
  }
}

int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
  }
  return n;
}

// Pack W (FP64, n x np) into the swizzled B blocks of k_recon_umma: for
// N block nb and K chunk kc a (2 NB rows x 128 B) image with rows c < NB
// = hi(W[k, nb NB + c]) and rows NB + c = the lo part, k in the chunk.
__global__ void k_pack_w(const ReconItem* __restrict__ items, void* const* ptrs, const int* __restrict__ ival) {
  if (items[blockIdx.y].Wp == nullptr) return;
  RecPlan D;
  rec_plan(items, blockIdx.y, ptrs, ival, D);
  const long long per_blk = (long long)(2 * D.NB) * 32;
  const long long total = (long long)D.nnb * D.nkc * per_blk;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long blk = e / per_blk;
    const int w = (int)(e - blk * per_blk);
    const int nb = (int)(blk / D.nkc), kc = (int)(blk - (long long)nb * D.nkc);
    const int row = w / 32, kk = w % 32;          // row of the block image, K within the chunk
    const int cl = row < D.NB ? row : row - D.NB;
    const int kg = kc * kKC + kk, cg = nb * D.NB + cl;
    float x = 0.f;
    if (kg < D.n && cg < D.np) x = (float)D.W[(long long)kg * D.ldw + cg];
    const float h = tf32_hi(x);
    const float v = row < D.NB ? h : x - h;
    float* img = const_cast<float*>(D.Wp) + blk * per_blk;
    img[(swz(row, kk >> 2) >> 2) + (kk & 3)] = v;
  }
}

}  // namespace um

bool umma_supported(int chimax) { return chimax >= 1 && chimax <= 128; }

cudaError_t launch_leg_umma(const LegItem* items, int n_items, int chimax, void* const* ptrs, const int* ival,
                            int* err, unsigned long long wait_ns, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  if (!umma_supported(chimax)) return cudaErrorInvalidValue;
  const um::LegSmem P = um::leg_smem(chimax);
  if (P.stages < 2) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(um::k_leg_umma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P.total);
  if (e != cudaSuccess) return e;
  for (int i0 = 0; i0 < n_items; i0 += kMaxItems) {
    const int n = std::min(kMaxItems, n_items - i0);
    um::k_leg_umma<<<um::sm_count(), um::kThreads, P.total, s>>>(items + i0, n, chimax, ptrs, ival, err, wait_ns);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

size_t recon_packed_floats(int nmax) {
  // the N blocking depends on the live n' <= nmax: take the largest layout
  size_t blocks_n = 0;
  for (int np = 1; np <= nmax; ++np) {
    const int nnb = (np + 127) / 128;
    const int NB = um::round_up((np + nnb - 1) / nnb, 8);
    blocks_n = std::max(blocks_n, (size_t)nnb * NB);
  }
  const int nkc = (um::round_up(nmax, 8) + um::kKC - 1) / um::kKC;
  return blocks_n * nkc * 2 * 32;
}

cudaError_t launch_recon_umma(const ReconItem* items, int n_items, int chimax, void* const* ptrs,
                              const int* ival, int* err, unsigned long long wait_ns, cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  if (!umma_supported(chimax)) return cudaErrorInvalidValue;
  const um::RecSmem P = um::rec_smem();
  um::k_pack_w<<<dim3(64, n_items), 256, 0, s>>>(items, ptrs, ival);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(um::k_recon_umma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P.total);
  if (e != cudaSuccess) return e;
  for (int i0 = 0; i0 < n_items; i0 += kMaxItems) {
    const int n = std::min(kMaxItems, n_items - i0);
    um::k_recon_umma<<<um::sm_count(), um::kThreads, P.total, s>>>(items + i0, n, ptrs, ival, err, wait_ns);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_gram_umma(const GramLegItem* items, int n_items, int splits_max, int chimax,
                             void* const* ptrs, const int* ival, int* err, unsigned long long wait_ns,
                             cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  if (!umma_supported(chimax)) return cudaErrorInvalidValue;
  const um::GramSmem P = um::gram_smem(chimax);
  if (P.stages < 2) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(um::k_gram_umma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)P.total);
  if (e != cudaSuccess) return e;
  for (int i0 = 0; i0 < n_items; i0 += kMaxItems) {
    const int n = std::min(kMaxItems, n_items - i0);
    um::k_gram_umma<<<um::sm_count(), um::kGramThreads, P.total, s>>>(items + i0, n, splits_max, chimax, ptrs, ival,
                                                                   err, wait_ns);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pepo
