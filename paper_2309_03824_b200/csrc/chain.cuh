// Fused two-product chain  Out[M x N2] = (In[M x K1] P[K1 x r]) Q[N2 x r]^T (+ bias)  with the
// rank-r intermediate T[M x r] kept on chip (tensor memory -> bf16 -> shared memory), written to
// memory only when the caller asks for it (T_save).  The forward pass is the chain (X, V, U),
// the backward data pass is the chain (dY, U, V).
#pragma once
#include "common.cuh"

namespace lrd {

// What both chain kernels' estimates are made of (see launch_chain in lrd_api.cu): microseconds of `waves` rounds of blocks
// that each take ng1 stages of the first product at t1 and `chunks` chunks of the second with m2 of k-blocks and `epilogue`
// of stores, the stores of a chunk beside the next one's k-blocks.
inline double chain_us(double fixed, int64_t waves, double ng1, double t1, int64_t chunks, double m2, double epilogue) {
    return fixed + (double)waves * (ng1 * t1 + m2 + (double)(chunks - 1) * (m2 > epilogue ? m2 : epilogue) + epilogue) + 2.0 * (double)(waves - 1);
}

// Row length in bytes (= swizzle span) of the boxes a block's `cols` columns of P are loaded in.  A box costs the TMA unit its
// rows, however short they are: columns that fill no whole 64-wide boxes are loaded in boxes 64 wide all the same, whose last
// one brings columns that nobody multiplies, rather than in three to seven boxes of 32- or 64-byte rows.  768 -> 768 at r = 192
// (slices of 48), 4096 tokens: forward 9.01 -> 8.80 us, backward with V frozen 16.6 -> 16.2; other widths within 1 %.
inline int p_box_span(int cols) { return cols > 32 ? 128 : cols > 16 ? 64 : 32; }

struct ChainArgs {
    int64_t M, K1, r, N2;
    const void* In; int64_t ld_in;     // [M x K1]
    const void* P; int64_t ldp;        // [K1 x r]
    const void* Q; int64_t ldq;        // [N2 x r]
    const void* bias;                  // [N2] or nullptr
    void* Out; int64_t ld_out;         // [M x N2]
    void* T_save; int64_t ldt;         // [M x r] or nullptr
    void* T_rows = nullptr;            // the first t_cols columns of T in rows of any stride and alignment, instead of T_save
    int64_t ld_rows = 0; int t_cols = 0;
    lrd_dtype_t dtype;
    int sm_share = 0;                  // SMs this launch can count on when it runs beside others (0: all of them)
};

// Overrides of the launch shape for benchmarking sweeps: cluster size, k-blocks per phase-1 stage,
// phase-2 chunk width.  0 = automatic.  Not thread-safe against concurrent launches.
void chain_tuning(int C, int G1, int BN2);
bool chain_eligible(const ChainArgs& c);
// Estimated microseconds (only for eligible arguments).
double chain_estimate(const ChainArgs& c);
lrd_status_t chain_launch(const ChainArgs& c, cudaStream_t stream);

// The same chain on pairs of SMs (tcgen05 cta_group::2): a cluster of 2 S blocks owns 256 rows.  `layers` are
// n <= kChainMaxLayers independent layers of equal shape that run in one launch (gridDim.z).  Needs more than
// 128 rows and a rank that splits into S slices of whole 32-column groups.
constexpr int kChainMaxLayers = 4;
// Overrides for sweeps and tests: pairs per cluster (1-4), k-blocks per phase-1 stage, phase-2 chunk width; 0 = automatic.
void chain_pair_tuning(int S, int G1, int BN2);
bool chain_pair_eligible(const ChainArgs* layers, int n);
double chain_pair_estimate(const ChainArgs* layers, int n);
lrd_status_t chain_pair_launch(const ChainArgs* layers, int n, cudaStream_t stream);

}  // namespace lrd
