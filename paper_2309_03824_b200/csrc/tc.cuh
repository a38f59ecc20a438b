// Internal interface of the tensor-core (tcgen05) kernels.
#pragma once
#include "common.cuh"

namespace lrd {

constexpr int kNumSms = 148;   // B200: tile and split choices are made against this count

// bf16, 16-byte aligned bases, leading dimensions multiples of 8 elements.
bool tc_gemm_eligible(const GemmArgs& g);
// fp32 partial-tile scratch a split product of this shape needs (0 when it is not split).
size_t tc_split_workspace_bytes(int64_t M, int64_t N, int64_t K);
// Unsplit product with a bf16 result on the persistent kernel (one block per SM walks over the tiles, the
// epilogue of a tile overlaps the MMAs of the next).  A K-major; no column sums.
lrd_status_t tc_gemm_persistent(const GemmArgs& g, cudaStream_t stream);
double tc_gemm_persistent_estimate(int64_t M, int64_t N, int64_t K);
// Estimated microseconds of a data product on the kernel tc_gemm would take for it (whole: without a split of the reduction),
// and whether it would split it.
double tc_gemm_estimate(int64_t M, int64_t N, int64_t K, bool whole = false);
bool tc_splits_data_product(int64_t M, int64_t N, int64_t K);
void tc_gemm_persistent_force_pairs(int blocks_per_mma);     // 0: automatic; 1 or 2: forced where the shape allows
// Weight gradients (both operands MN-major), up to kMaxWgrads of them in one launch.  Estimated microseconds on pairs of
// SMs (1e300 where that does not apply); all of them on pairs; all of them the fastest way (partials: scratch of each,
// which may be shared).
constexpr int kMaxWgrads = 8;
// Test hooks of the calling host thread: weight gradients on `blocks` blocks per MMA (1: single SMs, 2: pairs; 0: automatic) with
// tiles of `columns`, the reduction split over `split` blocks or pairs of a cluster; split data products likewise.  A product
// that no kernel runs in the form asked for is LRD_ERR_UNSUPPORTED.
struct WgradForm { int blocks, columns, split; };
WgradForm& tc_wgrad_form();
void tc_data_split_form(int columns, int split);
double tc_wgrad_pair_estimate(const GemmArgs* g, int n);
lrd_status_t tc_wgrad_pair(const GemmArgs* g, int n, cudaStream_t stream);       // (in the form of the test hook where that asks for pairs)
bool tc_wgrads_any_rows(const GemmArgs* g, int n);             // whether these are as well stored to rows of any alignment
lrd_status_t tc_wgrads(const GemmArgs* g, int n, float* const* partials, const size_t* partial_bytes, cudaStream_t stream);
// allow_split: a weight gradient (both operands MN-major), whose reduction may be split over blocks; else a data product (A
// K-major, no column sums).
lrd_status_t tc_gemm(const GemmArgs& g, bool allow_split, float* partials, size_t partial_bytes, cudaStream_t stream);

}  // namespace lrd
