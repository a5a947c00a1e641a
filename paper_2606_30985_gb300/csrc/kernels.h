// Launch wrappers of the libpepo kernels (host-callable, internal API).
#pragma once
#include "common.cuh"

namespace pepo {

// ---- k_tensor.cu (storage type T = float or double) ----------------------
template <typename T>
cudaError_t launch_leg_contract(const LegItem* items, int n_items, int chimax, void* const* ptrs, const int* ival,
                                cudaStream_t s);
template <typename T>
cudaError_t launch_copy(const TView* items, const int* out_refs, int n_items, int grid_x,
                        void* const* ptrs, const int* ival, cudaStream_t s);
template <typename T>
cudaError_t launch_gram_rows(const GramRowsItem* items, int n_items, int tiles_max, int splits_max,
                             int sym, void* const* ptrs, const int* ival, cudaStream_t s);
cudaError_t launch_gram_rows_reduce(const GramRowsItem* items, int n_items, int fmax,
                                    int splits_max, int sym, const int* ival, cudaStream_t s);
// exact FP32 Gram of the items whose branch value is `pass` (FP32 storage):
// four launches; acct as in launch_hh_extract
constexpr int kGramExactLaunches = 4;
cudaError_t launch_gram_exact(const GramRowsItem* items, int n_items, int fmax, int pass, void* const* ptrs,
                              const int* ival, double* acct, cudaStream_t s);
// kernels that launch_gram_leg enqueues (one per band of F up to chimax), and that the
// launchers with a limit on the items of a launch do
int gram_leg_launches(int chimax);
constexpr int kMaxItems = 512;
__host__ inline int item_launches(int n_items) { return (n_items + kMaxItems - 1) / kMaxItems; }
template <typename T>
cudaError_t launch_gram_leg(const GramLegItem* items, int n_items, int splits_max, int chimax,
                            void* const* ptrs, const int* ival, cudaStream_t s);
// canonical <-> stored site layout (perm[k] = canonical leg at layout position k)
template <typename T>
cudaError_t launch_permute(const void* in, void* out, int nlegs, const int* dims_canon, const int* perm,
                           int to_layout, cudaStream_t s);
// sum of the per-split partials; sym = 1 symmetrises the sum as (S + S^T) / 2
// rows: the split rule's rows per split (gram_leg_splits_k)
cudaError_t launch_gram_leg_reduce(const GramLegItem* items, int n_items, int chimax,
                                   int splits_max, int rows, int sym, const int* ival, cudaStream_t s);
template <typename T>
cudaError_t launch_reconstruct(const ReconItem* items, int n_items, int chimax, void* const* ptrs, const int* ival,
                               cudaStream_t s);
template <typename T>
cudaError_t launch_vec_contract(const VecItem* items, int n_items, void* const* ptrs, const int* ival, cudaStream_t s);
template <typename T>
cudaError_t launch_vec_pair(const VecPairItem* items, int n_items, void* const* ptrs, const int* ival, cudaStream_t s);

// ---- k_umma.cu (FP32 storage, TF32x3 on tcgen05 tensor cores, chi <= 128)
bool umma_supported(int chimax);
// err: device int; bit 0 is set when a pipeline wait of the kernel ran
// longer than wait_ns (the kernel then leaves its loops, lets its own MMAs and
// copies in flight finish, frees its tensor memory and returns), bit 1 when a
// reconstruct item has no packed-W workspace, bit 2 when one of those exit
// drains itself ran out of time
cudaError_t launch_leg_umma(const LegItem* items, int n_items, int chimax, void* const* ptrs, const int* ival,
                            int* err, unsigned long long wait_ns, cudaStream_t s);
// floats of the packed W workspace of one reconstruct item for n, n' <= nmax
size_t recon_packed_floats(int nmax);
// psi_new = psi W into the next layout (Q-less reconstruct), W from the bond core
cudaError_t launch_recon_umma(const ReconItem* items, int n_items, int chimax, void* const* ptrs,
                              const int* ival, int* err, unsigned long long wait_ns, cudaStream_t s);
// writes per-split partial sums S; the reduction with sym = 1 returns (S + S^T) / 2
cudaError_t launch_gram_umma(const GramLegItem* items, int n_items, int splits_max, int chimax,
                             void* const* ptrs, const int* ival, int* err, unsigned long long wait_ns,
                             cudaStream_t s);

// Split count shared by the Gram kernels and their reductions.
__host__ __device__ inline int gram_rows_splits(long long K, int splits_max) {
  long long s = (K + 511) / 512;
  if (s < 1) s = 1;
  return (int)(s < splits_max ? s : splits_max);
}
// split count of a free-leg Gram from its summed extent K = O * Q, about `rows`
// terms per split.  Tensor cores: 2048, 64 chunks of their pipeline.  SIMT in FP64:
// 512, so that the Grams of small bonds (K = 2048 at chi = 8) still spread over several
// SMs (the FP64 pipe of one needs 30 us for such a Gram alone); in FP32 2048, as a
// split also costs the sums of its groups (20 of 41 thousand clocks at chi = 20 with
// 512 terms).
constexpr int kGramLegRowsUmma = 2048;
__host__ __device__ constexpr int gram_leg_rows_simt(size_t item_bytes) { return item_bytes == 8 ? 512 : 2048; }
__host__ __device__ inline int gram_leg_splits_k(long long K, int splits_max, int rows) {
  long long s = K / rows;
  if (s < 1) s = 1;
  return (int)(s < splits_max ? s : splits_max);
}

}  // namespace pepo
