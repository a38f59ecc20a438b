// Tensor-core matrix product for sm_100a: TMA -> shared memory (128-byte swizzle) ->
// tcgen05.mma with the accumulator in tensor memory -> tcgen05.ld epilogue.
//
//   C[M x N] = op(A) op(B) (+ bias), bf16 in, fp32 accumulate, bf16 out.  The reduction dimension
//   may be split over gridDim.z (weight gradients reduce over all tokens but have few output tiles):
//     cluster split   the z blocks of a tile form a thread-block cluster; each block stages its fp32
//                     partial tile in shared memory, sends every peer the column slice that peer owns
//                     (bulk DSMEM copies) and adds the slices it receives in rank order -- one launch,
//                     no partials in global memory, a fixed order of additions;
//     global split    fp32 partial tiles in scratch memory that a second kernel adds in a fixed order
//                     (tiles wider than the cluster path supports, or more splits than a cluster holds).
//   No floating-point atomics anywhere: weight gradients are bit-reproducible.
//
// One 128 x BN output tile per block.  Warp 0 issues the TMA loads of the A operand and warp 6 those of the
// B operand (issuing a copy costs a thread about a hundred clocks, and an MN-major operand takes one copy per
// 64 columns: one warp alone issues a 40 KB stage in about 0.4 us, less than the memory system delivers),
// warp 1 owns tensor memory and issues the MMAs, warps 2-5 read the accumulator (each its own quarter of the
// 128 lanes) and store.  The single-thread instructions are issued under elect.sync by a converged warp.  Weight
// gradients have both operands MN-major (row / column index contiguous), data products A K-major (reduction index contiguous)
// and B either way: no product of the forward or backward pass needs a transposed copy.
//
// CONV: the filter gradient of a k x k convolution, dG[o][tap][i] = sum_p dout[p][o] in[p stride + tap - pad][i], is
// the same product with the taps side by side as columns (a tap takes whole 64-column blocks): A = dout[pixels x co],
// and a block of B is 64 consecutive output pixels' input channels at one tap, fetched by TMA in im2col mode.  The
// reduction runs over all pixels whatever the image size.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "conv.cuh"
#include "ptx.cuh"
#include "tc.cuh"
#include "tma.cuh"

namespace lrd {
namespace {

using namespace ptx;

constexpr int BM = 128, BK = 64;
constexpr int kThreads = 224;                         // warp 6: second TMA producer (the B operand)
constexpr int kMaxClusterSplits = 8;                 // portable cluster size

// ONES: every stage carries one more 64-wide MN-major block of B that holds 1.0 everywhere and is never
// overwritten; with N = BN + 16 the MMA then also forms sum_k A(m, k) in accumulator column BN (the bias
// gradient falls out of the dU product: its A operand is dY).
// G: 64-deep k-blocks per stage.  Two for the narrow tiles, whose MMAs take no longer than what a stage costs the issuing
// warp beside them (see tc_gemm_persistent.cu).  One with the ones block: two leave three stages of 64 KB, and the first MMA
// waits for twice the bytes (768 x 192 over 4096 tokens with the bias gradient 8.06 us with two, 7.88 with one; in clusters of
// two as the two-call backward runs it 10.78 / 10.36; over 9000 tokens, 264 x 264, the same).
template <int BN, bool ONES = false> struct Cfg {
    static constexpr int G = BN <= 128 && !ONES ? 2 : 1;
    static constexpr uint32_t A_STAGE_BYTES = G * BM * BK * 2;
    static constexpr uint32_t B_STAGE_BYTES = G * (BN * BK * 2 + (ONES ? 8192 : 0));
    static constexpr uint32_t STAGE_BYTES = A_STAGE_BYTES + B_STAGE_BYTES;
    static constexpr int STAGES_RAW = (200 * 1024) / STAGE_BYTES;
    static constexpr int STAGES = STAGES_RAW > 8 ? 8 : STAGES_RAW;
    // cluster split: fp32 staging tile + receive slots of the same size (+ column-sum slots), over the dead ring
    static constexpr uint32_t REDUCE_BYTES = BN <= 192 ? 2u * 128u * BN * 4u + 512u * (kMaxClusterSplits + 1) : 0u;
    static constexpr uint32_t RING_BYTES = STAGES * STAGE_BYTES;
    static constexpr uint32_t SMEM_BYTES = (RING_BYTES > REDUCE_BYTES ? RING_BYTES : REDUCE_BYTES) + 1024;   // + slack for 1024-B alignment
    static constexpr uint32_t TMEM_COLS = (BN + (ONES ? 32 : 0)) <= 64 ? 64 : ((BN + (ONES ? 32 : 0)) <= 128 ? 128 : 256);
};

struct TcParams {
    int64_t M, N;
    int64_t ldp;        // leading dimension of the fp32 partial tiles (N rounded up to 4)
    int kb_total, kb_per_split;
    void* C;            // bf16 [M x N] (ldc) or fp32 partials [splits][M x N] packed
    int64_t ldc;
    const __nv_bfloat16* bias;
    int partial;        // 1: write fp32 partials
    int cluster_splits; // > 1: the gridDim.z blocks of a tile are one cluster and reduce through shared memory
    // CONV: input channels, 64-column blocks of a tap and of all taps, k of the k x k taps, output grid, stride, pad
    int cv_ci, cv_nkc, cv_nblk, cv_k, cv_Ho, cv_Wo, cv_stride, cv_pad;
    // Operands that no launch of the same call still in flight writes are loaded before this launch's turn (griddepcontrol.wait)
    int a_early, b_early;
    int has_c_map;      // the result goes out by TMA
    float* colsum_partial;        // ONES, split: [splits][M] partial sums over k of A
    __nv_bfloat16* colsum_out;    // ONES, not split: [M]
    unsigned int* timeout_flag;
};

// What one launch computes: a product, or NP independent ones (weight gradients) whose row tiles follow one another in
// gridDim.y; every product takes the tile width and the cluster size of the launch.
template <int NP> struct TcLaunch {
    int row0[NP];       // first row tile of each product (INT_MAX: none)
    TcParams p[NP];
    CUtensorMap tA[NP], tB[NP], tC[NP];        // tC: boxes of 32 rows x 64 columns (tiles of one block) or one block's columns (cluster split, ADD)
};

// CONV: column of dG (= tap * ci + channel) that column `col` of the product belongs to; -1: padding
__device__ __forceinline__ int conv_col(const TcParams& p, int col) {
    const int blk = col / 64, c = (blk % p.cv_nkc) * 64 + col % 64;
    return blk < p.cv_nblk && c < p.cv_ci ? (blk / p.cv_nkc) * p.cv_ci + c : -1;
}

// kAdd: C += the product rounded to bf16 (fp32 sum, one more rounding) instead of C = it; column sums too.  A variant of its own:
// as a flag that every launch tests, its code stands between the stores of all of them, and a launch behind another kernel
// fetches it cold.  Backward passes in a graph, flag / variant: 768 -> 768 at rank 192, 4096 tokens, V frozen 18.05 / 17.33 us;
// 1024 -> 4096 at 512, 1021 tokens 23.7 / 22.7; 768 -> 3072 at 384, 600 tokens 18.95 / 18.10.
// kRows: C's rows have any stride and alignment.
constexpr int kStore = 0, kAdd = 1, kRows = 2;
template <int BN, bool A_MN, bool B_MN, bool ONES = false, bool CONV = false, int NP = 1, int OUT = kStore>
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_kernel(const __grid_constant__ TcLaunch<NP> L) {
    int prod = 0;
#pragma unroll
    for (int i = 1; i < NP; ++i)
        if ((int)blockIdx.y >= L.row0[i]) prod = i;
    const CUtensorMap &tmA = L.tA[prod], &tmB = L.tB[prod], &tmC = L.tC[prod];
    const TcParams p = L.p[prod];
    if (NP > 1 && (int64_t)blockIdx.x * BN >= p.N) {               // (the whole cluster: its blocks share x and y)
        griddep_wait();
        return;
    }
    static_assert(!ONES || (A_MN && B_MN && BN <= 192), "the ones block rides on an MN-major B of at most 192 columns");
    constexpr bool ADD = OUT == kAdd, ROWS = OUT == kRows;
    static_assert(OUT == kStore || !CONV, "only weight gradients");
    static_assert(!CONV || (A_MN && B_MN && !ONES && BN <= 192), "the filter gradient: both operands MN-major, split over a cluster or not at all");
    using C = Cfg<BN, ONES>;
    constexpr int STAGES = C::STAGES, G = C::G;
    constexpr uint32_t A_STAGE_BYTES = C::A_STAGE_BYTES, kBox = 8192u * G;        // MN-major box: 64 G k rows x 64 columns
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], acc_bar, red_bar;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const AbortCtx ab{&abort_flag, p.timeout_flag};
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    const int m0 = ((int)blockIdx.y - (NP > 1 ? L.row0[prod] : 0)) * BM, n0 = blockIdx.x * BN;
    const bool with_colsum = ONES && blockIdx.x == 0 && (NP == 1 || p.colsum_out);
    const int kb_begin = blockIdx.z * p.kb_per_split;
    const int kb_end = min(kb_begin + p.kb_per_split, p.kb_total);

    if (threadIdx.x == 0) {
        abort_flag = 0;
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        if (p.has_c_map) prefetch_tmap(&tmC);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        mbar_init(smem_u32(&acc_bar), 1);
        mbar_init(smem_u32(&red_bar), 1);
        if (p.cluster_splits > 1) {                        // bytes the peers will send this block
            const uint32_t S = (uint32_t)p.cluster_splits;
            uint32_t tx = (S - 1u) * 128u * (BN / S) * 4u;
            if (with_colsum && cluster_ctarank() == 0) tx += (S - 1u) * 512u;
            mbar_expect_tx(smem_u32(&red_bar), tx);
        }
        fence_mbar_init();
    }
    if (ONES) {          // bf16 1.0 in every element of the extra block of each stage
        for (uint32_t off = threadIdx.x * 16u; off < STAGES * kBox; off += kThreads * 16u)
            st_shared_v4(smem_base + (off / kBox) * C::STAGE_BYTES + A_STAGE_BYTES + BN * 128u * G + (off % kBox), 0x3F803F80u,
                         0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
        fence_proxy_async_smem();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_base_slot), C::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    // set-up above touched only this block's own shared and tensor memory: it may overlap the tail of the
    // previous kernel in the stream, and so may the loads of early operands (GemmArgs::a_early); everything else that touches global
    // memory stands behind the wait.
    // Every wait with a limit starts behind griddepcontrol.wait, as the launch in front, which may be the caller's, takes what time
    // it likes; with early operands it is a data pass of the same call, and the waits that need nothing of it start at once.
    const bool all_early = A_MN && p.a_early && p.b_early;
    if (!A_MN) griddep_wait();         // (in this order: see GemmArgs::a_early)
    griddep_launch_dependents();

    if (warp == 0) {
        // TMA producer: the whole warp runs the loop, one elected lane issues (operands stay uniform)
        if (!p.a_early) griddep_wait();
        int it = 0;
        for (int kb = kb_begin; kb < kb_end; kb += G, ++it) {          // (a k-block past this block's share is loaded, not multiplied)
            const int s = it % STAGES;
            const uint32_t ph = (it / STAGES) & 1;
            if (!mbar_wait_uniform(smem_u32(&empty_bar[s]), ph ^ 1, ab)) break;
            const uint32_t fb = smem_u32(&full_bar[s]);
            const uint32_t a_dst = smem_base + s * C::STAGE_BYTES;
            const int k0 = kb * BK;
            if (elect_one()) {
                mbar_expect_tx(fb, A_STAGE_BYTES + G * BN * BK * 2);   // the whole stage: warp 6's copies complete on the same barrier
                if (A_MN) {
#pragma unroll
                    for (int j = 0; j < BM / 64; ++j) tma_load_2d(a_dst + j * kBox, &tmA, fb, m0 + 64 * j, k0);
                } else {
#pragma unroll
                    for (int g = 0; g < G; ++g) tma_load_2d(a_dst + g * (BM * BK * 2), &tmA, fb, k0 + g * BK, m0);
                }
            }
            __syncwarp();
        }
        if (p.cluster_splits > 1) { cluster_arrive(); cluster_wait(); cluster_arrive_relaxed(); }   // barriers 1 and 2, see the epilogue
    } else if (warp == 6) {
        // second TMA producer: the B operand of every stage (its bytes are counted by warp 0's expect_tx; a copy that
        // lands before that arrival only makes the barrier's byte count negative for a moment)
        if (!p.b_early) griddep_wait();
        int it = 0;
        for (int kb = kb_begin; kb < kb_end; kb += G, ++it) {
            const int s = it % STAGES;
            const uint32_t ph = (it / STAGES) & 1;
            if (!mbar_wait_uniform(smem_u32(&empty_bar[s]), ph ^ 1, ab)) break;
            const uint32_t fb = smem_u32(&full_bar[s]);
            const uint32_t b_dst = smem_base + s * C::STAGE_BYTES + A_STAGE_BYTES;
            const int k0 = kb * BK;
            if (CONV) {
                // 64 G output pixels from pixel k0 on; a column block = 64 channels at one tap (blocks past the last tap load
                // the last one again, their columns are never stored)
                const int w = (k0 % p.cv_Wo) * p.cv_stride - p.cv_pad, hh = (k0 / p.cv_Wo) % p.cv_Ho, im = k0 / (p.cv_Wo * p.cv_Ho);
                if (elect_one()) {
#pragma unroll
                    for (int j = 0; j < BN / 64; ++j) {
                        const int blk = min(n0 / 64 + j, p.cv_nblk - 1), tap = blk / p.cv_nkc;
                        tma_load_im2col(b_dst + j * kBox, &tmB, fb, (blk % p.cv_nkc) * 64, w, hh * p.cv_stride - p.cv_pad, im,
                                        (uint32_t)(tap % p.cv_k), (uint32_t)(tap / p.cv_k));
                    }
                }
            } else if (elect_one()) {
                if (B_MN) {
#pragma unroll
                    for (int j = 0; j < BN / 64; ++j) tma_load_2d(b_dst + j * kBox, &tmB, fb, n0 + 64 * j, k0);
                } else {
#pragma unroll
                    for (int g = 0; g < G; ++g) tma_load_2d(b_dst + g * (BN * BK * 2), &tmB, fb, k0 + g * BK, n0);
                }
            }
            __syncwarp();
        }
        if (p.cluster_splits > 1) { cluster_arrive(); cluster_wait(); cluster_arrive_relaxed(); }
    } else if (warp == 1) {
        // MMA issuer: converged warp, elect.sync around the issue
        const uint32_t idesc = idesc_bf16(BN + (with_colsum ? 16 : 0), A_MN, B_MN);
        const uint64_t a_desc0 = A_MN ? smem_desc_sw128(smem_base, kBox, 1024) : smem_desc_sw128(smem_base, 0, 1024);
        const uint64_t b_desc0 = B_MN ? smem_desc_sw128(smem_base + A_STAGE_BYTES, kBox, 1024) : smem_desc_sw128(smem_base + A_STAGE_BYTES, 0, 1024);
        if (A_MN && !all_early) griddep_wait();
        int s = 0;
        uint32_t ph = 0, ready = kb_begin < kb_end ? mbar_test_wait(smem_u32(&full_bar[0]), 0) : 0u;
        bool ok = true;
        for (int kb = kb_begin; kb < kb_end; kb += G) {
            ok = mbar_wait_peeked(ready, smem_u32(&full_bar[s]), ph, ab);
            if (!ok) break;
            tc_fence_after();
            const uint64_t ad = a_desc0 + (uint32_t)s * (C::STAGE_BYTES >> 4), bd = b_desc0 + (uint32_t)s * (C::STAGE_BYTES >> 4);
            const uint32_t eb = smem_u32(&empty_bar[s]);
            if (++s == STAGES) { s = 0; ph ^= 1; }
            ready = kb + G < kb_end ? mbar_test_wait(smem_u32(&full_bar[s]), ph) : 0u;
            if (elect_one()) {
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if (g > 0 && kb + g >= kb_end) break;
#pragma unroll
                    for (int kk = 0; kk < BK / 16; ++kk)
                        mma_bf16_ss(tmem_base, ad + (A_MN ? (g * 4 + kk) * 128u : g * (BM * BK * 2 >> 4) + kk * 2u),
                                    bd + (B_MN ? (g * 4 + kk) * 128u : g * (BN * BK * 2 >> 4) + kk * 2u), idesc, g > 0 || kk > 0 ? 1u : (kb > kb_begin ? 1u : 0u));
                }
                mma_commit(eb);
            }
            __syncwarp();
        }
        if (ok && elect_one()) mma_commit(smem_u32(&acc_bar));
        __syncwarp();
        if (p.cluster_splits > 1) { cluster_arrive(); cluster_wait(); cluster_arrive_relaxed(); }
    } else if (p.cluster_splits > 1) {
        // ---- cluster split: reduce the partial tiles of the cluster's blocks through shared memory ----
        const int quarter = warp % 4;
        const int row = quarter * 32 + lane;
        const uint32_t S = (uint32_t)p.cluster_splits, self = cluster_ctarank();
        const uint32_t cs = BN / S;                        // columns this block owns (multiple of 8)
        const uint32_t chunk_bytes = 128u * cs * 4u, ngrp = cs / 4u;
        const uint32_t stage_base = smem_base, recv_base = smem_base + 128u * BN * 4u;
        const uint32_t cs_stage = recv_base + 128u * BN * 4u, cs_recv = cs_stage + 512u;
        if (A_MN && (ADD || !all_early)) griddep_wait();
        bool ok = mbar_wait_warp(smem_u32(&acc_bar), 0, ab);
        tc_fence_after();
        // barrier 1: this block's pipeline ring is dead (all its MMAs have completed).  Progress only: what the peers
        // must see of this block (its initialised barriers) is released by the arrivals of warps 0 and 1.
        cluster_arrive_relaxed();
        if (ok) {
            // partial tile -> staging, laid out [owner][row][cs] so that each owner's slice is one contiguous range
            const bool has_work = kb_begin < kb_end;       // a block past the end of the reduction contributes zeros
            // within a row of a slice the 16-byte groups are rotated by the row index: rows a power of two
            // apart in bytes would otherwise all hit the same banks
            const uint32_t rot = (uint32_t)row % ngrp;
            uint32_t grp = 0, dst_row = stage_base + (uint32_t)row * cs * 4u;   // group within the slice, row of the current owner's slice
#pragma unroll 1
            for (int c = 0; c < BN / 32; ++c) {
                uint32_t v[32];
                if (has_work) {
                    tmem_ld_32x32(tmem_base + ((uint32_t)(quarter * 32) << 16) + c * 32, v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = 0u;
                }
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    uint32_t rg = grp + rot;
                    if (rg >= ngrp) rg -= ngrp;
                    st_shared_v4(dst_row + rg * 16u, v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
                    if (++grp == ngrp) { grp = 0; dst_row += chunk_bytes; }
                }
            }
            if (with_colsum) {
                uint32_t cv[16];
                if (has_work) {
                    tmem_ld_32x16(tmem_base + ((uint32_t)(quarter * 32) << 16) + BN, cv);
                    tmem_ld_wait();
                } else {
                    cv[0] = 0u;
                }
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(cs_stage + (uint32_t)row * 4u), "r"(cv[0]) : "memory");
            }
        }
        fence_proxy_async_smem();
        tc_fence_before();
        cluster_wait();        // barrier 1 complete: every peer's ring is dead, its receive slots may be written
        ok = named_bar_and(2, 128, ok);
        if (warp == 2) {
            if (ok && elect_one()) {
                for (uint32_t t = 1; t < S; ++t) {
                    const uint32_t peer = (self + t) % S;
                    dsmem_bulk_copy(recv_base + self * chunk_bytes, stage_base + peer * chunk_bytes, chunk_bytes, smem_u32(&red_bar), peer);
                }
                if (with_colsum && self != 0) dsmem_bulk_copy(cs_recv + self * 512u, cs_stage, 512u, smem_u32(&red_bar), 0);
            }
            __syncwarp();
        }
        if (ok) {
            bool got = false;
            if (lane == 0) got = mbar_wait_cluster(smem_u32(&red_bar), 0, ab);
            ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
            if (ok) { for (int i = 0; i < 64 && !mbar_try_wait_cluster(smem_u32(&red_bar), 0); ++i) {} }
        }
        cluster_arrive_relaxed();   // barrier 2: everything addressed to this block has landed (progress only, no data)
        if (ok) {
            // this block's column slice: add the S partials in rank order, round once, store
            const int64_t grow = (int64_t)m0 + row;
            const int64_t gcol0 = (int64_t)n0 + self * cs;
            const uint32_t rot = (uint32_t)row % ngrp;
            // 8 columns of this row: the S partials in rank order (+ bias), rounded once
            auto sum8 = [&](uint32_t c4, uint32_t (&w)[4], float (&acc)[8]) {
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e] = 0.f;
                uint32_t g0 = c4 / 4u + rot, g1 = c4 / 4u + 1u + rot;
                if (g0 >= ngrp) g0 -= ngrp;
                if (g1 >= ngrp) g1 -= ngrp;
#pragma unroll 2
                for (uint32_t k = 0; k < S; ++k) {
                    const uint32_t row_base = (k == self ? stage_base + self * chunk_bytes : recv_base + k * chunk_bytes) + (uint32_t)row * cs * 4u;
                    float4 x, y;
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(row_base + g0 * 16u));
                    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(y.x), "=f"(y.y), "=f"(y.z), "=f"(y.w) : "r"(row_base + g1 * 16u));
                    acc[0] += x.x; acc[1] += x.y; acc[2] += x.z; acc[3] += x.w;
                    acc[4] += y.x; acc[5] += y.y; acc[6] += y.z; acc[7] += y.w;
                }
                const int64_t col = gcol0 + c4;
                if (p.bias) {
                    for (int e = 0; e < 8; ++e)
                        if (col + e < p.N) acc[e] += __bfloat162float(p.bias[col + e]);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) w[e] = pack_bf16(acc[2 * e], acc[2 * e + 1]);
            };
            auto store8 = [&](uint32_t c4, const uint32_t (&w)[4], const float (&acc)[8]) {
                const int64_t col = gcol0 + c4;
                if (grow >= p.M || col >= p.N) return;
                const int64_t at = CONV ? conv_col(p, (int)col) : col;        // (CONV: 8 columns are inside or outside together)
                if (CONV && at < 0) return;
                __nv_bfloat16* dst = (__nv_bfloat16*)p.C + grow * p.ldc + at;
                if (CONV || col + 8 <= p.N) {
                    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
                } else {
                    for (int e = 0; e < 8; ++e)
                        if (col + e < p.N) dst[e] = __float2bfloat16_rn(acc[e]);
                }
            };
            // 16 columns (one whole 32-byte sector) per store instruction where the layout allows, else two 16-byte stores
            const bool sectors = (p.ldc % 16 == 0) && (((uintptr_t)p.C & 31u) == 0) && (gcol0 % 16 == 0) && (!CONV || p.cv_ci % 16 == 0);
            const uint32_t slab = recv_base + self * chunk_bytes + (uint32_t)row * cs * 2u;        // (ADD; nobody sends to the own slot)
            for (uint32_t c4 = 0; c4 < cs; c4 += 16) {
                uint32_t w0[4], w1[4];
                float a0[8], a1[8];
                sum8(c4, w0, a0);
                const bool second = c4 + 8 < cs;
                if (second) sum8(c4 + 8, w1, a1);
                if (ADD || ROWS) {
                    st_shared_v4(slab + c4 * 2u, w0[0], w0[1], w0[2], w0[3]);
                    if (second) st_shared_v4(slab + c4 * 2u + 16u, w1[0], w1[1], w1[2], w1[3]);
                    continue;
                }
                const int64_t col = gcol0 + c4;
                if (sectors && second && grow < p.M && col + 16 <= p.N) {
                    const int64_t at = CONV ? conv_col(p, (int)col) : col;
                    if (CONV && at < 0) continue;
                    __nv_bfloat16* dst = (__nv_bfloat16*)p.C + grow * p.ldc + at;
                    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                                 ::"l"(dst), "r"(w0[0]), "r"(w0[1]), "r"(w0[2]), "r"(w0[3]), "r"(w1[0]), "r"(w1[1]), "r"(w1[2]), "r"(w1[3]) : "memory");
                } else {
                    store8(c4, w0, a0);
                    if (second) store8(c4 + 8, w1, a1);
                }
            }
            if (ROWS) {
                __syncwarp();
                const uint32_t rows0 = recv_base + self * chunk_bytes + quarter * 32u * cs * 2u;
                for (uint32_t c = 2u * lane; c < cs; c += 64u)
                    for (int r = 0; r < 32; r += 8)
                        store_any_rows8([&](int i) { return rows0 + (uint32_t)(r + i) * cs * 2u + c * 2u; }, (int)(p.M - (m0 + quarter * 32 + r) < 8 ? p.M - (m0 + quarter * 32 + r) : 8),
                                        (__nv_bfloat16*)p.C + (int64_t)(m0 + quarter * 32 + r) * p.ldc + gcol0 + c, p.ldc, (int)(p.N - gcol0 - c));
            }
            if (ADD) {
                fence_proxy_async_smem();
                __syncwarp();
                if (elect_one()) {
                    if (m0 + quarter * 32 < p.M && gcol0 < p.N) tma_add_2d(&tmC, recv_base + self * chunk_bytes + quarter * 32u * cs * 2u, (int)gcol0, m0 + quarter * 32);
                    tma_store_commit();
                    tma_store_wait_read<0>();
                }
                __syncwarp();
            }
            if (with_colsum && self == 0 && p.colsum_out && grow < p.M) {
                float t = 0.f;
                for (uint32_t k = 0; k < S; ++k) {
                    const uint32_t src = (k == 0 ? cs_stage : cs_recv + k * 512u) + (uint32_t)row * 4u;
                    float x;
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(src));
                    t += x;
                }
                if (ADD) add_into_bf16(p.colsum_out + grow, t);
                else p.colsum_out[grow] = __float2bfloat16_rn(t);
            }
        }
    } else {
        const int quarter = warp % 4;                      // lanes [32 q, 32 q + 32) of tensor memory
        if (A_MN && (ADD || !all_early)) griddep_wait();
        const bool ready = mbar_wait_warp(smem_u32(&acc_bar), 0, ab);
        tc_fence_after();
        if (ready) {
            const uint32_t lane_addr = tmem_base + ((uint32_t)(quarter * 32) << 16);
            const int64_t row = (int64_t)m0 + quarter * 32 + lane;
            const bool row_ok = row < p.M;
            if (with_colsum) {                             // accumulator column BN = sum over k of A(row, k)
                uint32_t cs[16];
                tmem_ld_32x16(lane_addr + BN, cs);
                tmem_ld_wait();
                if (row_ok) {
                    if (p.partial) p.colsum_partial[(int64_t)blockIdx.z * p.M + row] = __uint_as_float(cs[0]);
                    else if (ADD && p.colsum_out) add_into_bf16(p.colsum_out + row, __uint_as_float(cs[0]));
                    else if (p.colsum_out) p.colsum_out[row] = __float2bfloat16_rn(__uint_as_float(cs[0]));
                }
            }
            if (p.partial) {
#pragma unroll 1
                for (int c = 0; c < BN / 32; ++c) {
                    uint32_t v[32];
                    tmem_ld_32x32(lane_addr + c * 32, v);
                    tmem_ld_wait();
                    const int64_t col0 = (int64_t)n0 + c * 32;
                    if (!row_ok || col0 >= p.N) continue;
                    float* dst = (float*)p.C + ((int64_t)blockIdx.z * p.M + row) * p.ldp + col0;
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        if (col0 + g * 4 + 4 <= p.N) {
                            *reinterpret_cast<uint4*>(dst + g * 4) = make_uint4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
                        } else {
                            for (int e = 0; e < 4; ++e)
                                if (col0 + g * 4 + e < p.N) dst[g * 4 + e] = __uint_as_float(v[4 * g + e]);
                        }
                    }
                }
            } else {
                // 64 columns of the warp's 32 rows at a time through a slab of their own in the dead ring (128-byte swizzle), then
                // out by one TMA store, or, ADD, by one that adds in L2 (the fp32 sum of two bf16 values, rounded once).  Stores
                // straight from the registers, each lane a row of its own, were four dependent steps of scattered 16-byte
                // accesses, and reading C for them as many trips to memory: 4096 x 512 over 1021 tokens, accumulating, 128 blocks
                // 128 wide: 6 us behind the last MMA, the pass 41.9 us, now 37.0; 768 x 192 over 128 tokens, a pass 19.0 -> 18.5.
                const uint32_t slab0 = smem_base + (uint32_t)quarter * (BN / 64 * 4096u), row_off = (uint32_t)lane * 128u, row_xor = (uint32_t)lane & 7u;
#pragma unroll 1
                for (int c = 0; c < BN / 64; ++c) {
                    const int col0 = n0 + c * 64;
                    if (col0 >= p.N && !CONV) break;       // (uniform)
                    uint32_t v[64];
                    tmem_ld_32x32(lane_addr + c * 64, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
                    tmem_ld_32x32(lane_addr + c * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
                    tmem_ld_wait();
                    uint32_t w[32];
#pragma unroll
                    for (int e = 0; e < 32; ++e) w[e] = pack_bf16(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
                    if (CONV) {                            // 8 columns of one tap, inside or outside together
#pragma unroll
                        for (int g = 0; g < 8; ++g) {
                            const int at = col0 < p.N ? conv_col(p, col0 + g * 8) : -1;
                            if (row_ok && at >= 0)
                                *reinterpret_cast<uint4*>((__nv_bfloat16*)p.C + row * p.ldc + at) = make_uint4(w[4 * g], w[4 * g + 1], w[4 * g + 2], w[4 * g + 3]);
                        }
                        continue;
                    }
                    const uint32_t slab = slab0 + (uint32_t)c * 4096u;
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        st_shared_v4(slab + row_off + (((uint32_t)g ^ row_xor) << 4), w[4 * g], w[4 * g + 1], w[4 * g + 2], w[4 * g + 3]);
                    if (ROWS) {              // rows that TMA cannot address: a row at a time, a lane two columns
                        __syncwarp();
                        for (int r = 0; r < 32; r += 8)
                            store_any_rows8([&](int i) { return slab + (uint32_t)(r + i) * 128u + ((((uint32_t)lane >> 2) ^ (uint32_t)i) << 4) + ((uint32_t)lane & 3u) * 4u; },
                                            (int)(p.M - (m0 + quarter * 32 + r) < 8 ? p.M - (m0 + quarter * 32 + r) : 8),
                                            (__nv_bfloat16*)p.C + (int64_t)(m0 + quarter * 32 + r) * p.ldc + col0 + 2 * lane, p.ldc, (int)(p.N - col0 - 2 * lane));
                        continue;
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (elect_one()) {
                        if (m0 + quarter * 32 < p.M) {
                            if (ADD) tma_add_2d(&tmC, slab, col0, m0 + quarter * 32);
                            else tma_store_2d(&tmC, slab, col0, m0 + quarter * 32);
                        }
                        tma_store_commit();
                    }
                    __syncwarp();
                }
                tma_store_wait_read<0>();                  // shared memory may go once the stores have read it
                __syncwarp();
            }
        }
    }

    griddep_wait();        // (early loads: this launch ends no sooner than the one before it, on which the launches behind it rely)
    // cluster split, barrier 2: no block leaves while a peer may still be reading its slice out of this
    // block's shared memory
    if (p.cluster_splits > 1) cluster_wait();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (abort_flag) {            // give copies and MMAs still in flight time to land before freeing
            for (int i = 0; i < 256; ++i) __nanosleep(1000);
        }
        tc_fence_after();
        tmem_dealloc(tmem_base, C::TMEM_COLS);
    }
}

// out[m][n] = sum_z partial[z][m][n], z ascending; 4 columns per thread.
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const float* __restrict__ partial, int splits, int64_t M,
                                                            int64_t N, int64_t ldp,
                                                            __nv_bfloat16* __restrict__ C, int64_t ldc,
                                                            const float* __restrict__ colsum_partial,
                                                            __nv_bfloat16* __restrict__ colsum_out, int add) {
    const int64_t n4 = (N + 3) / 4;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= M * n4) {                                // trailing threads: the column sums, one row each
        const int64_t m = idx - M * n4;
        if (colsum_out && m < M) {
            float t = 0.f;
            for (int z = 0; z < splits; ++z) t += colsum_partial[(int64_t)z * M + m];
            if (add) add_into_bf16(colsum_out + m, t);
            else colsum_out[m] = __float2bfloat16_rn(t);
        }
        return;
    }
    const int64_t m = idx / n4, n = (idx % n4) * 4;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    const bool full = n + 4 <= N;
    for (int z = 0; z < splits; ++z) {
        const float* src = partial + ((int64_t)z * M + m) * ldp + n;
        if (full) {
            const float4 v = *reinterpret_cast<const float4*>(src);
            acc[0] += v.x; acc[1] += v.y; acc[2] += v.z; acc[3] += v.w;
        } else {
            for (int e = 0; e < 4; ++e)
                if (n + e < N) acc[e] += src[e];
        }
    }
    for (int e = 0; e < 4; ++e)
        if (n + e < N) {
            if (add) add_into_bf16(C + m * ldc + n + e, acc[e]);
            else C[m * ldc + n + e] = __float2bfloat16_rn(acc[e]);
        }
}

template <int BN, bool A_MN, bool B_MN, bool ONES = false, bool CONV = false, int NP = 1, int OUT = kStore>
lrd_status_t launch(const TcLaunch<NP>& L, dim3 grid, cudaStream_t stream, bool wait_ahead = true) {
    auto kern = tc_gemm_kernel<BN, A_MN, B_MN, ONES, CONV, NP, OUT>;
    const TcParams& p = L.p[0];
    static bool configured_on[kMaxDevices] = {};     // per instantiation; the attribute is sticky per function
    bool& configured = configured_on[device_slot()];
    if (!configured) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN, ONES>::SMEM_BYTES) != cudaSuccess)
            return LRD_ERR_CUDA;
        configured = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = Cfg<BN, ONES>::SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = p.cluster_splits > 1 ? (unsigned)p.cluster_splits : 1u;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the kernel waits (griddepcontrol.wait) for all but early operands
    attr[1].val.programmaticStreamSerializationAllowed = wait_ahead ? 1 : 0;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, kern, L) != cudaSuccess) return LRD_ERR_CUDA;
    count_launch();
    return LRD_OK;
}

int out_mode(const GemmArgs& g, bool scratch) { return scratch ? kStore : g.add ? kAdd : g.any_rows ? kRows : kStore; }

template <int BN, bool ONES, int NP = 1>
lrd_status_t launch_wgrad(int out, const TcLaunch<NP>& L, dim3 grid, cudaStream_t s, bool wait_ahead = true) {
    return out == kAdd    ? launch<BN, true, true, ONES, false, NP, kAdd>(L, grid, s, wait_ahead)
           : out == kRows ? launch<BN, true, true, ONES, false, NP, kRows>(L, grid, s, wait_ahead)
                          : launch<BN, true, true, ONES, false, NP>(L, grid, s, wait_ahead);
}

inline bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// Tensor map of the result where it leaves by TMA, and the early operands.
bool result_map(const GemmArgs& g, bool add, int bn, int cluster, bool partial, CUtensorMap* t, TcParams* p) {
    p->has_c_map = !partial && !g.any_rows && (cluster <= 1 || add);
    p->a_early = g.a_early; p->b_early = g.b_early;
    return !p->has_c_map || make_tmap_2d_bf16(t, g.C, (uint64_t)g.M, (uint64_t)g.N, (uint64_t)g.ldc, 32, cluster > 1 ? (uint32_t)(bn / cluster) : 64u, cluster <= 1);
}

uint32_t stage_kblocks(int bn, bool ones) {
    switch (bn) {
        case 64:  return ones ? Cfg<64, true>::G : Cfg<64>::G;
        case 128: return ones ? Cfg<128, true>::G : Cfg<128>::G;
        default:  return 1;
    }
}
static_assert(Cfg<192>::G == 1 && Cfg<192, true>::G == 1 && Cfg<256>::G == 1, "stage_kblocks");

}  // namespace

bool tc_gemm_eligible(const GemmArgs& g) {
    if (g.dtype != LRD_BF16 || g.M < 1 || g.N < 1 || g.K < 1) return false;
    if (g.M > (int64_t)65535 * BM || g.K > (int64_t)1 << 30 || g.N > (int64_t)1 << 30) return false;
    if (!aligned16(g.A) || !aligned16(g.B) || (!aligned16(g.C) && !g.any_rows)) return false;
    if (g.lda % 8 || g.ldb % 8 || (g.ldc % 8 && !g.any_rows)) return false;
    return true;
}

// Tile width.  Every MMA of a tile reads its 128 x 16 block of A from shared memory whatever its width, and
// every tile streams its own copy of A, so a narrow tile pays the same A traffic for fewer columns: below
// about 154 columns the cost of a k-block is taken as constant, above as proportional to the width.
// The reduction is split until the machine is full -> minimise tiles x per-tile cost.
static int pick_bn(int64_t M, int64_t N) {
    const int64_t mt = (M + BM - 1) / BM;
    int best = 64;
    double best_cost = 1e300;
    for (int bn : {256, 192, 128, 64}) {
        if (bn == 64 && N > 64) continue;
        const double cost = (double)(mt * ((N + bn - 1) / bn)) * (bn < 154 ? 154.0 : (double)bn);
        if (cost < best_cost) { best_cost = cost; best = bn; }
    }
    return best;
}

static int global_splits(int64_t M, int64_t N, int64_t K, int bn) {
    const int64_t tiles = ((M + BM - 1) / BM) * ((N + bn - 1) / bn);
    const int64_t kb = (K + BK - 1) / BK;
    int64_t s = kNumSms / tiles;
    if (s < 1) s = 1;
    if (s > kb / 4) s = kb / 4;          // at least four k-blocks per split
    if (s < 1) s = 1;
    if (s > 64) s = 64;
    // no empty split: shrink until every z has work
    const int64_t per = (kb + s - 1) / s;
    s = (kb + per - 1) / per;
    return (int)s;
}

// Clusters of S blocks that can be resident at once (S blocks need S free SMs inside one GPC, so this is
// fewer than SMs / S).  All instantiations hold one block per SM, so one of them answers for all.
static int max_active_clusters(int S) {
    static int cache_on[kMaxDevices][kMaxClusterSplits + 1] = {};
    int* cache = cache_on[device_slot()];
    if (S < 2 || S > kMaxClusterSplits) return kNumSms;
    if (cache[S] == 0) {
        auto kern = tc_gemm_kernel<64, true, true, false>;
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1, 1, (unsigned)S);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = Cfg<64, false>::SMEM_BYTES;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 1;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = (unsigned)S;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<64, false>::SMEM_BYTES) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
            cudaGetLastError();
            n = (kNumSms - 20) / S;                     // no answer (no device yet): a cautious guess
        }
        cache[S] = n;
    }
    return cache[S];
}

// How a product whose reduction may be split is run.
struct SplitPlan {
    int bn;
    int cluster;     // > 1: cluster split (blocks per tile)
    int global;      // > 1: global split (partials in scratch memory + reduce kernel)
};

// Estimated microseconds of weight gradients in one launch: `tiles` of 128 x bn, each in a cluster of S blocks (1: waves of
// single blocks), `deepest` k-blocks in the longest share and `kblocks` in all.  A block's time is its operand traffic (every
// block streams its share of A and B through one SM's memory port, all together through what L2 delivers), and a split adds
// the exchange, which grows with the tile.  Measured / estimated: 3072 x 384 over 4096 tokens (192 wide, 2 blocks) 14.8 / 15.3;
// over 16384 40.8 / 40.4; 768 x 192 over 4096 (64, 4) 7.1 / 6.7; 1536 x 384 over 2048 (192, 4) 9.4 / 9.1; 4096 x 256 over 8192
// (128, 2) 19.9 / 18.9.  Short reductions and many tiles are better left whole (no exchange): 3072 x 384 over 4096 tokens 14.9 us
// in clusters of 2, 12.5 in 144 blocks 64 wide; over 512 6.8 / 5.1; 1536 x 384 over 2048 9.6 / 7.0.  Many waves want wide tiles:
// 4096 x 4096 over 8192 tokens, 64 / 128 / 192 wide 426 / 299 / 274 us (without L2's limit the 128 wide ones looked best), 274 on
// pairs; 4096 x 1024 115 / 74 / 90, on pairs 63.
static double split_us(int bn, int S, int64_t tiles, int64_t deepest, int64_t kblocks) {
    const double kb_bytes = BM * BK * 2.0 + bn * BK * 2.0;
    if (S > 1) return 4.2 + 0.022 * (bn - 64) + std::max(0.7e6 * (double)deepest * kb_bytes / 110e9, 0.8e6 * (double)kblocks * kb_bytes / 14e12);
    // single blocks: the issue loop's or the MMAs' pace, or, once every SM has a block, what L2 delivers to all of them
    const int64_t waves = (tiles + kNumSms - 1) / kNumSms;
    const double pace = std::max({0.2, 0.0017 * bn, (double)std::min<int64_t>(tiles, kNumSms) * kb_bytes / 18.5e6});
    return 2.5 + 0.006 * (bn - 64) + (double)(waves * deepest) * pace + 3.0 * (double)(waves - 1);
}

// One weight gradient: the candidates are tile widths that the reduction buffers fit (<= 192) and cluster sizes that divide
// the tile into slices of whole 16-byte groups; where no cluster per tile fits, single blocks or shares through scratch memory.
// A launch that runs beside a data chain (clusters of at most 2) gets some 50 SMs: few wide blocks, always split, leave most
// of them to others (step of a block of 768-wide layers, U frozen: 182 us with the plans of a launch that runs alone, 178.5 so).
static SplitPlan pick_split(int64_t M, int64_t N, int64_t K, bool ones, int max_cluster = 0, double* us = nullptr) {
    const int top = max_cluster >= 2 && max_cluster < kMaxClusterSplits ? max_cluster : kMaxClusterSplits;
    const int64_t mt = (M + BM - 1) / BM, kb = (K + BK - 1) / BK;
    SplitPlan best{pick_bn(M, N), 1, 1};
    if (ones && best.bn > 192) best.bn = 192;
    best.global = global_splits(M, N, K, best.bn);
    const int64_t tiles0 = mt * ((N + best.bn - 1) / best.bn), share = (kb + best.global - 1) / best.global;
    double best_t = split_us(best.bn, 1, tiles0 * best.global, share, 0) + (best.global > 1 ? 8.0 + 8e6 * (double)(best.global * M * N) / 5e12 : 0.0);     // + partials out and in, one more launch
    for (int bn : {192, 128, 64}) {
        const int64_t nt = (N + bn - 1) / bn, tiles = mt * nt;
        if (nt * bn >= N + 64 && bn > 64) continue;              // a narrower width covers N with less waste
        for (int S = top; S >= 1; --S) {
            if (bn % (8 * S) || S > kb || (S == 1 && top == 2)) continue;
            if (S > 1 && tiles > max_active_clusters(S)) continue;     // one wave: a second wave would double the time
            const int64_t per = (kb + S - 1) / S;
            double t = split_us(bn, S, tiles, per, tiles * S * per);
            if (top == 2) t = 3.0 + 0.8e6 * std::max((double)per * (BM + bn) * 128.0 / 110e9, (double)(tiles * S * per) * (BM + bn) * 128.0 / 11.5e12) + bn / 120.0;
            if (t < best_t) { best_t = t; best.bn = bn; best.cluster = S; best.global = 1; }
        }
    }
    if (us) *us = best_t;
    return best;
}

WgradForm& tc_wgrad_form() {
    static thread_local WgradForm form{0, 0, 0};
    return form;
}
static thread_local int t_data_columns = 0, t_data_split = 0;
void tc_data_split_form(int columns, int split) { t_data_columns = columns; t_data_split = split; }

// A data product with few tiles and a long reduction (a short batch through a wide layer) is the latency of one tile's
// k-blocks: about 0.13 us each for the narrow tiles such products run on, after some 3.3 us of launch, first loads and
// epilogue.  Split over the blocks of a cluster it is a share of them and the exchange: 128 tokens, 3072 -> 384 9.4 us
// on the persistent kernel, 5.4 us split eight ways; 768 -> 384 4.4 us, where a split would not be faster.
static bool split_data_product(int64_t M, int64_t N, int64_t K, SplitPlan* out, double* us) {
    const int64_t mt = (M + BM - 1) / BM, kb = (K + BK - 1) / BK;
    double best = 3.3 + 0.13 * (double)kb;
    bool found = false;
    if (t_data_columns) {
        *us = best;
        *out = SplitPlan{t_data_columns, t_data_split, 1};
        return true;
    }
    for (int bn : {64, 128}) {
        const int64_t tiles = mt * ((N + bn - 1) / bn);
        for (int S = kMaxClusterSplits; S >= 2; S /= 2) {
            if (tiles > max_active_clusters(S) || S > kb) continue;
            const double t = 4.6 + 0.13 * (double)((kb + S - 1) / S) + 0.006 * (bn - 64);
            if (t < 0.95 * best) { best = t; *out = SplitPlan{bn, S, 1}; found = true; }
            break;
        }
    }
    *us = best;
    return found;
}

bool tc_splits_data_product(int64_t M, int64_t N, int64_t K) {
    SplitPlan sp;
    double us;
    return split_data_product(M, N, K, &sp, &us);
}

double tc_gemm_estimate(int64_t M, int64_t N, int64_t K, bool whole) {
    SplitPlan sp;
    double us;
    return !whole && split_data_product(M, N, K, &sp, &us) ? us : tc_gemm_persistent_estimate(M, N, K);
}

// fp32 partial tiles [splits][M][ldp], then (for the optional column sums) [splits][M]; nothing for a cluster split
size_t tc_split_workspace_bytes(int64_t M, int64_t N, int64_t K) {
    size_t need = 0;
    for (int v = 0; v < 4; ++v) {                    // with and without the column sums, for either cluster limit
        const int ones = v & 1;
        const int s = pick_split(M, N, K, ones != 0, (v & 2) ? 2 : 0).global;
        const size_t n = s > 1 ? align_up((size_t)s * M * ((N + 3) / 4 * 4) * sizeof(float), 256) + align_up((size_t)s * M * sizeof(float), 256) : 0;
        need = need > n ? need : n;
    }
    return need;
}

lrd_status_t tc_gemm(const GemmArgs& g, bool allow_split, float* partials, size_t partial_bytes,
                     cudaStream_t stream) {
    if (!tc_gemm_eligible(g)) return LRD_ERR_UNSUPPORTED;
    const bool ones = g.a_colsum != nullptr;
    int splits = 1, cluster, bn;
    if (allow_split) {                                     // weight gradients
        if (!g.a_mn_major || !g.b_mn_major || g.bias) return LRD_ERR_UNSUPPORTED;        // (only data products add a bias)
        double us;
        const WgradForm& form = tc_wgrad_form();
        const int64_t n = g.any_rows ? (g.N + 15) / 16 * 16 : g.N;          // (scratch was asked for at the padded rank)
        const SplitPlan sp = form.blocks ? SplitPlan{form.columns, form.split, 1} : pick_split(g.M, n, g.K, ones, g.max_cluster_split, &us);
        // pairs where the tiles leave no room for a cluster per tile
        if (form.blocks ? form.blocks == 2 : tc_wgrad_pair_estimate(&g, 1) < 0.95 * us) return tc_wgrad_pair(&g, 1, stream);
        bn = sp.bn; cluster = sp.cluster; splits = sp.global;
    } else {                                               // data products: the persistent kernel, or a split of the reduction
        if (g.a_mn_major || ones) return LRD_ERR_UNSUPPORTED;
        SplitPlan dp;
        double us;
        if (g.whole || !split_data_product(g.M, g.N, g.K, &dp, &us)) return tc_gemm_persistent(g, stream);
        bn = dp.bn; cluster = dp.cluster;
    }
    const int64_t ldp = (g.N + 3) / 4 * 4;
    const size_t tile_bytes = align_up((size_t)splits * g.M * ldp * sizeof(float), 256);
    if (splits > 1 && (!partials || partial_bytes < tile_bytes + (ones ? (size_t)splits * g.M * sizeof(float) : 0)))
        return LRD_ERR_WORKSPACE;
    const int kb_total = (int)((g.K + BK - 1) / BK);
    const int zdim = cluster > 1 ? cluster : splits;
    const int kb_per = (kb_total + zdim - 1) / zdim;

    TcLaunch<1> L{};
    CUtensorMap &tA = L.tA[0], &tB = L.tB[0];
    const uint32_t kbox = BK * stage_kblocks(bn, ones);             // k rows of an MN-major box
    bool ok = g.a_mn_major ? make_tmap_2d_bf16(&tA, g.A, (uint64_t)g.K, (uint64_t)g.M, (uint64_t)g.lda, kbox, 64)
                           : make_tmap_2d_bf16(&tA, g.A, (uint64_t)g.M, (uint64_t)g.K, (uint64_t)g.lda, BM, BK);
    ok = ok && (g.b_mn_major ? make_tmap_2d_bf16(&tB, g.B, (uint64_t)g.K, (uint64_t)g.N, (uint64_t)g.ldb, kbox, 64)
                             : make_tmap_2d_bf16(&tB, g.B, (uint64_t)g.N, (uint64_t)g.K, (uint64_t)g.ldb, (uint32_t)bn, BK));
    TcParams& p = L.p[0];
    ok = ok && result_map(g, g.add && splits == 1, bn, cluster, splits > 1, &L.tC[0], &p);
    if (!ok) return LRD_ERR_CUDA;

    p.M = g.M; p.N = g.N; p.ldp = ldp; p.kb_total = kb_total; p.kb_per_split = kb_per;
    p.partial = splits > 1 ? 1 : 0;
    p.cluster_splits = cluster;
    p.timeout_flag = device_timeout_flag();
    p.C = splits > 1 ? (void*)partials : g.C;
    p.ldc = g.ldc;
    p.bias = (const __nv_bfloat16*)g.bias;
    p.colsum_partial = (ones && splits > 1) ? (float*)((uint8_t*)partials + tile_bytes) : nullptr;
    p.colsum_out = (ones && splits == 1) ? (__nv_bfloat16*)g.a_colsum : nullptr;
    dim3 grid((unsigned)((g.N + bn - 1) / bn), (unsigned)((g.M + BM - 1) / BM), (unsigned)zdim);
    lrd_status_t st;
    const int out = out_mode(g, splits > 1);               // (shares through scratch memory: the second kernel adds)
    if (ones) {
        switch (bn) {
            case 192: st = launch_wgrad<192, true>(out, L, grid, stream, !g.in_turn); break;
            case 128: st = launch_wgrad<128, true>(out, L, grid, stream, !g.in_turn); break;
            default:  st = launch_wgrad<64, true>(out, L, grid, stream, !g.in_turn); break;
        }
    } else if (allow_split) {
        switch (bn) {
            case 256: st = launch_wgrad<256, false>(out, L, grid, stream, !g.in_turn); break;
            case 192: st = launch_wgrad<192, false>(out, L, grid, stream, !g.in_turn); break;
            case 128: st = launch_wgrad<128, false>(out, L, grid, stream, !g.in_turn); break;
            default:  st = launch_wgrad<64, false>(out, L, grid, stream, !g.in_turn); break;
        }
    } else if (bn == 128) {
        st = g.b_mn_major ? launch<128, false, true>(L, grid, stream) : launch<128, false, false>(L, grid, stream);
    } else {
        st = g.b_mn_major ? launch<64, false, true>(L, grid, stream) : launch<64, false, false>(L, grid, stream);
    }
    if (st != LRD_OK || splits == 1) return st;
    const int64_t work = g.M * ((g.N + 3) / 4) + (ones ? g.M : 0);
    splitk_reduce_kernel<<<(unsigned)((work + 255) / 256), 256, 0, stream>>>(
        partials, splits, g.M, g.N, ldp, (__nv_bfloat16*)g.C, g.ldc, p.colsum_partial,
        ones ? (__nv_bfloat16*)g.a_colsum : nullptr, g.add);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? LRD_OK : LRD_ERR_CUDA;
}

// Estimated microseconds of one launch for all of g's products, with one width and cluster size.
static double group_estimate(const GemmArgs* g, int n, int bn, int S) {
    int64_t tiles = 0, deepest = 0, kblocks = 0;
    for (int i = 0; i < n; ++i) {
        const int64_t t = ((g[i].M + BM - 1) / BM) * ((g[i].N + bn - 1) / bn), kb = ((g[i].K + BK - 1) / BK + S - 1) / S;
        tiles += t;
        deepest = std::max(deepest, kb);
        kblocks += t * S * kb;
    }
    return S > 1 && tiles > max_active_clusters(S) ? 1e300 : split_us(bn, S, tiles, deepest, kblocks);
}

// The fastest of them by that estimate.
static double best_group(const GemmArgs* g, int n, int* bn, int* S) {
    const int top = g[0].max_cluster_split >= 2 && g[0].max_cluster_split < kMaxClusterSplits ? g[0].max_cluster_split : kMaxClusterSplits;
    double us = 1e300;
    for (int b : {192, 128, 64})
        for (int c = top; c >= 1; --c) {
            if (b % (8 * c)) continue;
            const double t = group_estimate(g, n, b, c);
            if (t < us) { us = t; *bn = b; *S = c; }
        }
    return us;
}

constexpr double kNextLaunch = 2.0;            // a launch behind another one drains and fills the SMs anew

// Gradients whose rows TMA cannot address run on single SMs only: worth it where pairs would not save more than the launch that
// copies a padded result, some 3 us.  Over 360 backward passes of packed layers (64 to 8192 tokens, ranks 61 to 1001, each mask) the
// choice costs 0.3 % on average against the fastest measurement (always in place 0.5 %, always copied 7.0): 2048 tokens, 4096 -> 4096 at
// rank 250, nothing frozen, in place / copied 37.8 / 41.2 us; 4096 tokens, 4096 -> 4096 at rank 499 84.3 / 80.7.
bool tc_wgrads_any_rows(const GemmArgs* g, int n) {
    if (tc_wgrad_form().blocks) return false;
    double single = kNextLaunch * (n - 1), pairs = single;
    for (int i = 0; i < n; ++i) {
        double us;
        pick_split(g[i].M, g[i].N, g[i].K, g[i].a_colsum != nullptr, g[i].max_cluster_split, &us);
        single += us;
        pairs += std::min(us, tc_wgrad_pair_estimate(&g[i], 1));
    }
    if (n > 1) {
        int bn, S;
        single = std::min(single, best_group(g, n, &bn, &S));
        pairs = std::min(pairs, tc_wgrad_pair_estimate(g, n));
    }
    return single <= pairs + 3.0;
}

template <int BN, bool ONES>
static lrd_status_t launch_group(const GemmArgs* g, int n, int S, cudaStream_t stream) {
    TcLaunch<kMaxWgrads> L{};
    unsigned nx = 0, ny = 0;
    const uint32_t kbox = BK * Cfg<BN, ONES>::G;
    for (int i = 0; i < kMaxWgrads; ++i) {
        L.row0[i] = i < n ? (int)ny : INT_MAX;
        if (i >= n) continue;
        if (!make_tmap_2d_bf16(&L.tA[i], g[i].A, (uint64_t)g[i].K, (uint64_t)g[i].M, (uint64_t)g[i].lda, kbox, 64) ||
            !make_tmap_2d_bf16(&L.tB[i], g[i].B, (uint64_t)g[i].K, (uint64_t)g[i].N, (uint64_t)g[i].ldb, kbox, 64))
            return LRD_ERR_CUDA;
        TcParams& p = L.p[i];
        if (!result_map(g[i], g[i].add, BN, S, false, &L.tC[i], &p)) return LRD_ERR_CUDA;
        p.M = g[i].M; p.N = g[i].N; p.ldp = g[i].N;
        p.kb_total = (int)((g[i].K + BK - 1) / BK);
        p.kb_per_split = (p.kb_total + S - 1) / S;
        p.cluster_splits = S;
        p.timeout_flag = device_timeout_flag();
        p.C = g[i].C; p.ldc = g[i].ldc;
        p.colsum_out = (__nv_bfloat16*)g[i].a_colsum;
        nx = std::max(nx, (unsigned)((g[i].N + BN - 1) / BN));
        ny += (unsigned)((g[i].M + BM - 1) / BM);
    }
    return launch_wgrad<BN, ONES>(out_mode(g[0], false), L, dim3(nx, ny, (unsigned)S), stream, !g[0].in_turn);
}

// The weight gradients of one backward pass.  Each alone has few output tiles and one pays for its launch, its first loads and
// its exchange over a chip that is mostly idle, so as many as the caller has at hand go into one launch, on single SMs
// (a cluster per tile) or on pairs, when the estimate is below the sum of theirs.  Forward and backward of a layer with nothing
// frozen, each alone / together: 4096 -> 4096 at rank 512, 8192 tokens 189 / 182 us; rank 256 142 / 132; 768 -> 3072 at 384,
// 4096 tokens 73 / 62; 1024 -> 4096 at 512, 1024 tokens 48 / 42; 768 -> 768 at 192, 300 tokens 30 / 21.  Two launches cost 2 us
// more than their times alone (backward of the first layer at rank 1000, 2 x 64 tiles on pairs: two launches 256 us, one of two waves 242).
lrd_status_t tc_wgrads(const GemmArgs* g, int n, float* const* partials, const size_t* partial_bytes, cudaStream_t stream) {
    const WgradForm& form = tc_wgrad_form();
    bool ones = false, together = n > 1 && n <= kMaxWgrads;
    int64_t rows = 0;
    double separate = kNextLaunch * (n - 1);
    for (int i = 0; i < n && together; ++i) {
        together = tc_gemm_eligible(g[i]) && g[i].a_mn_major && g[i].b_mn_major && !g[i].bias && g[i].max_cluster_split == g[0].max_cluster_split &&
                   g[i].add == g[0].add && g[i].any_rows == g[0].any_rows;
        if (!together) break;
        ones = ones || g[i].a_colsum;
        rows += (g[i].M + BM - 1) / BM;
        double us;
        pick_split(g[i].M, g[i].N, g[i].K, g[i].a_colsum != nullptr, g[i].max_cluster_split, &us);
        separate += std::min(us, tc_wgrad_pair_estimate(&g[i], 1));
    }
    if (together && rows <= 65535) {
        int bn = 0, S = 1;
        double us = best_group(g, n, &bn, &S);
        if (!(us < separate)) { us = separate; bn = 0; }
        if (form.blocks) { bn = form.columns; S = form.split; }
        if (form.blocks ? form.blocks == 2 : tc_wgrad_pair_estimate(g, n) < us) return tc_wgrad_pair(g, n, stream);
        switch (bn) {
            case 192: return ones ? launch_group<192, true>(g, n, S, stream) : launch_group<192, false>(g, n, S, stream);
            case 128: return ones ? launch_group<128, true>(g, n, S, stream) : launch_group<128, false>(g, n, S, stream);
            case 64:  return ones ? launch_group<64, true>(g, n, S, stream) : launch_group<64, false>(g, n, S, stream);
            default:  break;
        }
    }
    for (int i = 0; i < n; ++i) {
        const lrd_status_t st = tc_gemm(g[i], true, partials[i], partial_bytes[i], stream);
        if (st != LRD_OK) return st;
    }
    return LRD_OK;
}

// Filter gradient (see CONV above): M = co, N = taps x 64-column blocks, K = output pixels.
lrd_status_t tc_conv_filter(const void* dout, const void* in, void* dG, int64_t B, const ConvGeom& g, int64_t ci, int64_t co,
                            bool a_early, bool b_early, cudaStream_t stream) {
    if (!tc_conv_eligible(B, g, ci, co, LRD_BF16, dout, in, dG)) return LRD_ERR_UNSUPPORTED;
    const int64_t P = B * g.Ho * g.Wo, taps = (int64_t)g.k * g.k, nkc = (ci + 63) / 64, N = taps * nkc * 64;
    SplitPlan sp = pick_split(co, N, P, true);             // (tiles of at most 192 columns)
    if (tc_wgrad_form().blocks == 1) sp = SplitPlan{tc_wgrad_form().columns, tc_wgrad_form().split, 1};
    if (sp.cluster < 2) sp.cluster = 1;                    // tiles enough to fill the GPU: each reduces over all pixels
    TcLaunch<1> L{};
    CUtensorMap &tA = L.tA[0], &tB = L.tB[0];
    const uint32_t kbox = BK * stage_kblocks(sp.bn, false);
    bool ok = make_tmap_2d_bf16(&tA, dout, (uint64_t)P, (uint64_t)co, (uint64_t)co, kbox, 64);
    ok = ok && make_tmap_im2col_bf16(&tB, in, (uint64_t)B, (uint64_t)g.H, (uint64_t)g.W, (uint64_t)ci, -g.pad, -g.pad, g.Ho, g.Wo, g.stride, kbox);
    if (!ok) return LRD_ERR_CUDA;
    TcParams& p = L.p[0];
    p.M = co; p.N = N; p.ldp = N;
    p.kb_total = (int)((P + BK - 1) / BK);
    p.kb_per_split = (p.kb_total + sp.cluster - 1) / sp.cluster;
    p.cluster_splits = sp.cluster;
    p.timeout_flag = device_timeout_flag();
    p.C = dG; p.ldc = taps * ci;
    p.a_early = a_early; p.b_early = b_early;
    p.cv_ci = (int)ci; p.cv_nkc = (int)nkc; p.cv_nblk = (int)(taps * nkc); p.cv_k = g.k;
    p.cv_Ho = g.Ho; p.cv_Wo = g.Wo; p.cv_stride = g.stride; p.cv_pad = g.pad;
    dim3 grid((unsigned)((N + sp.bn - 1) / sp.bn), (unsigned)((co + BM - 1) / BM), (unsigned)sp.cluster);
    switch (sp.bn) {
        case 192: return launch<192, true, true, false, true>(L, grid, stream);
        case 128: return launch<128, true, true, false, true>(L, grid, stream);
        default:  return launch<64, true, true, false, true>(L, grid, stream);
    }
}

}  // namespace lrd
