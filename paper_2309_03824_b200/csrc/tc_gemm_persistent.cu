// Persistent tensor-core matrix product for sm_100a (unsplit products with a bf16 result):
//   C[M x N] = A op(B) (+ bias), A K-major
// One block per SM walks over the 128 x BN output tiles (tile t -> row tile t % m_tiles, column tile
// t / m_tiles, so that blocks working at the same time share the B operand in L2).  The accumulator is
// double-buffered in tensor memory: while the eight epilogue warps round tile i to bf16 and store it
// (each warp 32-column pieces of its own 32 rows, through [32 x 32] shared-memory slabs and TMA stores that clip the ragged
// edges), the MMA warp already accumulates tile i + 1.  A short reduction (K of a few hundred, as in the
// second product of an unfused decomposed layer) is otherwise all epilogue.
// Warp 0: TMA producer.  Warp 1: tensor memory + MMA issue.  Warps 2-9: epilogue.  Single-thread
// instructions are issued under elect.sync by a converged warp; every wait is bounded.
//
// CG = 2 runs the same loop on pairs of blocks (a cluster of two SMs, tcgen05 cta_group::2): a pair owns a
// 256 x BN tile, each block loads its own 128 rows of A but only HALF of the B tile, and the even block
// issues MMAs of 256 rows that read both halves.  Per k-block a block then takes (16 KB + BN x 64 B)
// instead of (16 KB + BN x 128 B) through its L2 -> shared-memory path, which is what bounds the wide
// tiles: at BN = 256 the shared-memory port sees 64 KB (fill + operand reads) per 512 MMA cycles instead
// of 96 KB.
#include "common.cuh"
#include "ptx_pair.cuh"
#include "tc.cuh"
#include "tma.cuh"

namespace lrd {
namespace {

using namespace ptx;

constexpr int BM = 128, BK = 64;
constexpr int kThreads = 320;                                // TMA producer, MMA issuer, 8 x epilogue
constexpr uint32_t kATile = BM * BK * 2;
constexpr uint32_t kSlabBytes = 32 * 32 * 2;                 // one warp's slab: 32 rows x 32 columns of bf16
constexpr uint32_t kStagingBytes = 8 * 2 * kSlabBytes;

template <int BN, int CG> struct PCfg {
    static constexpr int BNH = BN / CG;                      // columns of B this block loads
    // 64-deep k-blocks per stage.  A stage costs the issuing warp some 250 clocks beside its MMAs (a wait, an election, a
    // commit); the four MMAs of a k-block of a narrow tile take no longer, so narrow tiles have two per stage.  One
    // 128-row tile, 3072 -> 384: 13.3 us with one k-block per stage and each stage's barrier first looked at when it is
    // needed, 10.7 with the look ahead, 9.1 with two k-blocks; pairs and wide tiles, paced by their MMAs and
    // loads, are 1 % slower with two.
    static constexpr int G = CG == 1 && BN <= 128 ? 2 : 1;
    static constexpr uint32_t B_TILE = BNH * BK * 2;
    static constexpr uint32_t STAGE_BYTES = G * (kATile + B_TILE);
    static constexpr int STAGES_RAW = (193 * 1024) / STAGE_BYTES;         // beside 32 KB of store slabs
    static constexpr int STAGES = STAGES_RAW > 8 ? 8 : STAGES_RAW;
    static constexpr uint32_t SMEM_BYTES = STAGES * STAGE_BYTES + kStagingBytes + 1024;
    static constexpr uint32_t TMEM_COLS = 2 * BN <= 128 ? 128 : (2 * BN <= 256 ? 256 : 512);
    static constexpr uint32_t BUF_COLS = TMEM_COLS / 2;      // column offset of the second accumulator
};

template <int CG>
__device__ __forceinline__ void load2d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int x, int y) {
    if (CG == 2) tma_load_2d_pair(dst, m, bar, x, y);        // bar: shared::cluster address (the even block's barrier)
    else tma_load_2d(dst, m, bar, x, y);
}

struct PParams {
    int64_t M, N;
    int kb_total, m_tiles, n_tiles;
    int b_early;              // the first stages' B is loaded before this launch's turn
    const __nv_bfloat16* bias;
    unsigned int* timeout_flag;
};

template <int BN, bool B_MN, int CG>
__global__ void __launch_bounds__(kThreads, 1)
tc_gemm_persistent_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                          const __grid_constant__ CUtensorMap tmC, const PParams p) {
    using C = PCfg<BN, CG>;
    constexpr int BNH = C::BNH;
    static_assert(CG == 1 || CG == 2, "blocks per MMA");
    static_assert(CG == 1 || !B_MN || BNH % 64 == 0, "an MN-major half of B is made of 64-column boxes");
    constexpr int STAGES = C::STAGES, G = C::G;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], out_full[2], out_empty[2];
    __shared__ __align__(16) uint16_t bias_s[2][256];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;

    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t staging_base = smem_base, ring_base = smem_base + kStagingBytes;
    const AbortCtx ab{&abort_flag, p.timeout_flag};
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    const int n_tiles_total = p.m_tiles * p.n_tiles;         // p.m_tiles counts row tiles of 128 CG rows
    const int h = CG == 2 ? (int)cluster_ctarank() : 0;      // this block's half of the pair
    const int unit = (int)blockIdx.x / CG, n_units = (int)gridDim.x / CG;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        prefetch_tmap(&tmC);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&out_full[i]), 1);
            mbar_init(smem_u32(&out_empty[i]), 8 * CG);       // the epilogue warps of every block of the pair
        }
        fence_mbar_init();
    }
    if (warp == 1) {
        if (CG == 2) {
            tmem_alloc_pair(smem_u32(&tmem_base_slot), C::TMEM_COLS);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(smem_u32(&tmem_base_slot), C::TMEM_COLS);
            tmem_relinquish();
        }
    }
    tc_fence_before();
    if (CG == 2) {                   // the other block's barriers exist before anything signals them
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    // A pair's loads all complete on the even block's barrier, which its MMA warp waits on.
    auto full = [&](int s) { return CG == 2 ? map_to_cta(smem_u32(&full_bar[s]), 0) : smem_u32(&full_bar[s]); };
    auto load_a = [&](int s, int kb, int m0, uint32_t fb) {
#pragma unroll
        for (int g = 0; g < G; ++g) load2d<CG>(ring_base + s * C::STAGE_BYTES + g * kATile, &tmA, fb, (kb + g) * BK, m0);
    };
    auto load_b = [&](int s, int kb, int n0, uint32_t fb) {
        const uint32_t b_dst = ring_base + s * C::STAGE_BYTES + G * kATile;
        if (B_MN) {
#pragma unroll
            for (int j = 0; j < BNH / 64; ++j) load2d<CG>(b_dst + j * (8192 * G), &tmB, fb, n0 + 64 * j, kb * BK);
        } else {
#pragma unroll
            for (int g = 0; g < G; ++g) load2d<CG>(b_dst + g * C::B_TILE, &tmB, fb, (kb + g) * BK, n0);
        }
    };
    // set-up above touched only this block's own shared and tensor memory: it may overlap the tail of the
    // previous kernel in the stream.  So may, where the call says so, the load of B for the first tile, as much as the ring holds
    // (see GemmArgs::b_early): what follows the wait is then the load of A alone.  Everything else that touches global memory stands
    // behind the wait.  Forward passes as two products, 72 shapes of 64 to 8192 tokens: 1.3 % on average, 1024 -> 4096 at rank 512,
    // 64 tokens 8.9 -> 8.6 us, 768 -> 3072 at 384, 512 tokens 9.5 -> 9.2; the one that loses is 1024 -> 4096 at 512 tokens, 10.65 -> 10.85.
    int early = 0;                                           // stages whose B is on its way
    if (!B_MN && p.b_early && warp == 0 && unit < n_tiles_total) {
        early = min(STAGES, (p.kb_total + G - 1) / G);
        if (elect_one())
            for (int s = 0; s < early; ++s) {
                if (h == 0) mbar_expect_tx(smem_u32(&full_bar[s]), CG * C::STAGE_BYTES);
                load_b(s, s * G, (unit / p.m_tiles) * BN + h * BNH, full(s));
            }
        __syncwarp();
    }
    griddep_wait();
    // (in this order: see GemmArgs::a_early; one warp of a block is enough, and the producer has its first loads to issue: 64 tokens,
    // 768 -> 3072 at rank 384, passes on a stream 8.33 -> 8.24 us)
    if (warp != 0) griddep_launch_dependents();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        int s = 0, kb0 = 0;
        uint32_t ph = 1;
        bool ok = true;
        if (early) {             // (apart from the loop below: tests in it took 3072 -> 768 at 384, 4096 tokens, from 20.5 to 20.9 us)
            if (elect_one())
                for (int i = 0; i < early; ++i) load_a(i, i * G, (unit % p.m_tiles) * (BM * CG) + h * BM, full(i));
            __syncwarp();
            kb0 = early * G;
            if (early < STAGES) s = early; else ph = 0;
        }
        for (int t = unit; t < n_tiles_total && ok; t += n_units) {
            const int m0 = (t % p.m_tiles) * (BM * CG) + h * BM, n0 = (t / p.m_tiles) * BN + h * BNH;
            for (int kb = kb0; kb < p.kb_total; kb += G) {       // k-blocks past the last read as zeros
                ok = mbar_wait_uniform(smem_u32(&empty_bar[s]), ph, ab);
                if (!ok) break;
                const uint32_t fb = full(s);
                if (elect_one()) {
                    if (h == 0) mbar_expect_tx(smem_u32(&full_bar[s]), CG * C::STAGE_BYTES);
                    load_a(s, kb, m0, fb);
                    load_b(s, kb, n0, fb);
                }
                __syncwarp();
                if (++s == STAGES) { s = 0; ph ^= 1; }
            }
            kb0 = 0;
        }
    } else if (warp == 1 && h == 0) {
        // ------------------------------------------------------------------ MMA issuer (the even block of a pair)
        constexpr uint32_t idesc = CG == 2 ? idesc_bf16_pair(BN, false, B_MN) : idesc_bf16(BN, false, B_MN);
        // the descriptors of a stage differ from these in the start address only (bits 0-13, in 16-byte units); a k-step of
        // 16 moves it by 2048 bytes (MN-major) or 32 (K-major: 32 within a k-block, then the next tile)
        const uint64_t a_desc0 = smem_desc_sw128(ring_base, 0, 1024);
        const uint64_t b_desc0 = B_MN ? smem_desc_sw128(ring_base + G * kATile, 8192 * G, 1024) : smem_desc_sw128(ring_base + G * kATile, 0, 1024);
        int s = 0, i = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int t = unit; t < n_tiles_total && ok; t += n_units, ++i) {
            const int buf = i & 1;
            const uint32_t d_tmem = tmem_base + (uint32_t)buf * C::BUF_COLS;
            ok = mbar_wait_uniform(smem_u32(&out_empty[buf]), ((i >> 1) & 1) ^ 1, ab);      // accumulator buffer drained
            uint32_t ready = mbar_test_wait(smem_u32(&full_bar[s]), ph);
            for (int kb = 0; kb < p.kb_total && ok; kb += G) {
                ok = mbar_wait_peeked(ready, smem_u32(&full_bar[s]), ph, ab);
                if (!ok) break;
                tc_fence_after();
                const uint64_t ad = a_desc0 + (uint32_t)s * (C::STAGE_BYTES >> 4), bd = b_desc0 + (uint32_t)s * (C::STAGE_BYTES >> 4);
                const uint32_t eb = smem_u32(&empty_bar[s]);
                const bool last = kb + G >= p.kb_total;
                if (++s == STAGES) { s = 0; ph ^= 1; }
                ready = last ? 0u : mbar_test_wait(smem_u32(&full_bar[s]), ph);
                if (elect_one()) {
#pragma unroll
                    for (int g = 0; g < G; ++g) {
                        if (g > 0 && kb + g >= p.kb_total) break;
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            const uint32_t ao = g * (kATile >> 4) + kk * 2u;
                            const uint32_t bo = B_MN ? (g * 4 + kk) * 128u : g * (C::B_TILE >> 4) + kk * 2u;
                            const uint32_t acc = g > 0 || kk > 0 ? 1u : (kb > 0 ? 1u : 0u);
                            if (CG == 2) mma_bf16_ss_pair(d_tmem, ad + ao, bd + bo, idesc, acc);
                            else mma_bf16_ss(d_tmem, ad + ao, bd + bo, idesc, acc);
                        }
                    }
                    if (CG == 2) {       // both blocks' stages are free, both blocks' accumulators are ready
                        mma_commit_pair(eb, 3);
                        if (last) mma_commit_pair(smem_u32(&out_full[buf]), 3);
                    } else {
                        mma_commit(eb);
                        if (last) mma_commit(smem_u32(&out_full[buf]));
                    }
                }
                __syncwarp();
            }
        }
    } else if (warp >= 2) {
        // ------------------------------------------------------------------ epilogue
        const int q = warp % 4;                              // tensor-memory lanes [32 q, 32 q + 32)
        const int hw = (warp - 2) / 4;                       // two warps share a quarter: they take alternate 32-column pieces
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t slab0 = staging_base + (uint32_t)(warp - 2) * 2u * kSlabBytes;
        const uint32_t row_off = (uint32_t)lane * 64u, row_xor = ((uint32_t)lane >> 1) & 3u;
        uint16_t next_bias[4];
        bias_fetch(next_bias, p.bias, (int64_t)(unit / p.m_tiles) * BN + 32 * hw, p.N);
        int i = 0, sb = 0;
        bool ok = true;
        for (int t = unit; t < n_tiles_total && ok; t += n_units, ++i) {
            const int buf = i & 1;
            const int m0 = (t % p.m_tiles) * (BM * CG) + h * BM, n0 = (t / p.m_tiles) * BN;
            const bool rows_inside = m0 + q * 32 < p.M;      // (uniform) a pair's odd block may hang over the last row tile
            ok = mbar_wait_uniform(smem_u32(&out_full[buf]), (i >> 1) & 1, ab);
            if (!ok) break;
            if (p.bias) bias_put(&bias_s[buf][32 * hw], next_bias, BN / 64);
            bias_fetch(next_bias, p.bias, (int64_t)((t + n_units) / p.m_tiles) * BN + 32 * hw, p.N);        // of the next tile
            tc_fence_after();
            const uint32_t d_tmem = lane_addr + (uint32_t)buf * C::BUF_COLS;
#pragma unroll 1
            for (int c0 = hw; c0 < BN / 32; c0 += 4) {       // this warp's pieces, two at a time
                if (n0 + c0 * 32 >= p.N) break;              // (uniform) nothing of this piece is inside C
                const bool second = c0 + 2 < BN / 32 && n0 + c0 * 32 + 64 < p.N;
                uint32_t v2[2][32];
                tmem_ld_32x32(d_tmem + c0 * 32, v2[0]);
                if (second) tmem_ld_32x32(d_tmem + c0 * 32 + 64, v2[1]);
                tmem_ld_wait();
#pragma unroll
                for (int h2 = 0; h2 < 2; ++h2, ++sb) {
                    if (h2 == 1 && !second) break;           // (uniform)
                    uint32_t (&v)[32] = v2[h2];
                    const int col0 = n0 + (c0 + 2 * h2) * 32;
                    if (p.bias) bias_add(v, &bias_s[buf][32 * c0 + 64 * h2]);
                    const uint32_t slab = slab0 + (uint32_t)(sb & 1) * kSlabBytes;
                    if (sb >= 2) {                           // the store that last read this slab has finished reading
                        tma_store_wait_read<1>();
                        __syncwarp();
                    }
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc)
                        st_shared_v4(slab + row_off + ((((uint32_t)cc) ^ row_xor) << 4),
                                     pack_bf16(__uint_as_float(v[8 * cc]), __uint_as_float(v[8 * cc + 1])),
                                     pack_bf16(__uint_as_float(v[8 * cc + 2]), __uint_as_float(v[8 * cc + 3])),
                                     pack_bf16(__uint_as_float(v[8 * cc + 4]), __uint_as_float(v[8 * cc + 5])),
                                     pack_bf16(__uint_as_float(v[8 * cc + 6]), __uint_as_float(v[8 * cc + 7])));
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (elect_one()) {
                        if (rows_inside) tma_store_2d(&tmC, slab, col0, m0 + q * 32);
                        tma_store_commit();
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                if (CG == 2) mbar_arrive_remote(smem_u32(&out_empty[buf]), 0);
                else mbar_arrive(smem_u32(&out_empty[buf]));
            }
        }
        tma_store_wait_read<0>();                            // shared memory may go once the stores have read it
        __syncwarp();
    }

    tc_fence_before();
    if (CG == 2) {
        // neither block leaves (or frees tensor memory) while the other may still signal one of its barriers,
        // read its shared memory with an MMA or write its accumulators: every thread of the pair is past all of
        // that when it arrives here
        cluster_arrive();
        cluster_wait();
    } else {
        __syncthreads();
    }
    if (warp == 1) {
        if (abort_flag) {            // give copies and MMAs still in flight time to land before freeing
            for (int i = 0; i < 256; ++i) __nanosleep(1000);
        }
        tc_fence_after();
        if (CG == 2) tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
        else tmem_dealloc(tmem_base, C::TMEM_COLS);
    }
}

template <int BN, bool B_MN, int CG>
lrd_status_t launch_p(const CUtensorMap& tA, const CUtensorMap& tB, const CUtensorMap& tC, const PParams& p, unsigned blocks,
                      cudaStream_t stream) {
    auto kern = tc_gemm_persistent_kernel<BN, B_MN, CG>;
    static bool configured_on[kMaxDevices] = {};     // per instantiation; the attribute is sticky per function
    bool& configured = configured_on[device_slot()];
    if (!configured) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, PCfg<BN, CG>::SMEM_BYTES) != cudaSuccess)
            return LRD_ERR_CUDA;
        configured = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = PCfg<BN, CG>::SMEM_BYTES;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the kernel waits (griddepcontrol.wait) for all but an early B
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = CG;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = CG == 2 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, kern, tA, tB, tC, p) != cudaSuccess) return LRD_ERR_CUDA;
    count_launch();
    return LRD_OK;
}

template <int BN, int CG>
lrd_status_t launch_p_major(bool b_mn, const CUtensorMap& tA, const CUtensorMap& tB, const CUtensorMap& tC, const PParams& p, unsigned blocks,
                            cudaStream_t s) {
    return b_mn ? launch_p<BN, true, CG>(tA, tB, tC, p, blocks, s) : launch_p<BN, false, CG>(tA, tB, tC, p, blocks, s);
}

// Tile shape.  Per k-block a block streams (A tile + its part of the B tile) from L2 at about 64 B/clk and
// its MMAs take 2 BN clocks; the slowest unit walks over ceil(tiles / units) tiles.  Minimise the product over
// the tile widths and over single blocks (148 units, 128-row tiles) and pairs (74 units, 256-row tiles);
// earlier candidates (wider, single) win ties.
struct PShape { int bn, cg; };
int g_force_cg = 0;                  // 0: by the cost above; 1 or 2: forced where possible (test hook)

PShape pick_shape_p(int64_t M, int64_t N) {
    if (N <= 64) return {64, 1};
    const int cands[4] = {256, 192, 128, 64};
    PShape best = {128, 1};
    double best_cost = 1e300;
    for (int cg = 1; cg <= 2; ++cg) {
        if (g_force_cg && cg != g_force_cg) continue;
        if (cg == 2 && M <= BM) continue;
        const int64_t mt = (M + BM * cg - 1) / (BM * cg);
        const int64_t units = kNumSms / cg;
        for (int bn : cands) {
            if (cg == 2 && bn != 256 && bn != 128) continue;
            const int64_t tiles = mt * ((N + bn - 1) / bn);
            const double fill = (double)(kATile + (bn / cg) * BK * 2) / 64.0, mma = 2.0 * bn;
            const double cost = (double)((tiles + units - 1) / units) * (fill > mma ? fill : mma);
            if (cost < best_cost) { best_cost = cost; best = {bn, cg}; }
        }
    }
    return best;
}

}  // namespace

// Estimated microseconds of one product (see launch_chain in lrd_api.cu): the k-blocks of a tile at the issue loop's, the
// tensor pipe's or the loads' pace, whichever is slowest; the epilogue of a tile beside the next tile's k-blocks.
double tc_gemm_persistent_estimate(int64_t M, int64_t N, int64_t K) {
    const PShape sh = pick_shape_p(M, N);
    const int64_t kb = (K + BK - 1) / BK, units = kNumSms / sh.cg;
    const int64_t tiles = ((M + BM * sh.cg - 1) / (BM * sh.cg)) * ((N + sh.bn - 1) / sh.bn), waves = (tiles + units - 1) / units;
    const double mma = 4.0 * (sh.bn / 2.0 > 32 + sh.bn / 4.0 ? sh.bn / 2.0 : 32 + sh.bn / 4.0) / 1965.0;
    const double load = (double)(kATile + sh.bn / sh.cg * BK * 2) * 6.6e-6, issue = sh.cg == 1 && sh.bn <= 128 ? 0.16 : 0.19;
    const double main = (double)kb * (mma > load ? (mma > issue ? mma : issue) : (load > issue ? load : issue)), epilogue = 0.0195 * sh.bn;
    return 1.7 + main + (double)(waves - 1) * (main > epilogue ? main : epilogue) + epilogue;
}

void tc_gemm_persistent_force_pairs(int cg) { g_force_cg = (cg == 1 || cg == 2) ? cg : 0; }

lrd_status_t tc_gemm_persistent(const GemmArgs& g, cudaStream_t stream) {
    if (!tc_gemm_eligible(g) || g.a_colsum || g.a_mn_major) return LRD_ERR_UNSUPPORTED;
    PShape sh = pick_shape_p(g.M, g.N);
    if (g_force_cg == 2 && sh.cg != 2) { g_force_cg = 0; sh = pick_shape_p(g.M, g.N); g_force_cg = 2; }
    const int bn = sh.bn, cg = sh.cg, bnh = bn / cg;
    CUtensorMap tA, tB, tC;
    const uint32_t kbox = BK * (cg == 1 && bn <= 128 ? 2 : 1);         // k rows of an MN-major box
    bool ok = make_tmap_2d_bf16(&tA, g.A, (uint64_t)g.M, (uint64_t)g.K, (uint64_t)g.lda, BM, BK);
    ok = ok && (g.b_mn_major ? make_tmap_2d_bf16(&tB, g.B, (uint64_t)g.K, (uint64_t)g.N, (uint64_t)g.ldb, kbox, 64)
                             : make_tmap_2d_bf16(&tB, g.B, (uint64_t)g.N, (uint64_t)g.K, (uint64_t)g.ldb, (uint32_t)bnh, BK));
    ok = ok && make_tmap_2d_bf16(&tC, g.C, (uint64_t)g.M, (uint64_t)g.N, (uint64_t)g.ldc, 32, 32);
    if (!ok) return LRD_ERR_CUDA;
    PParams p;
    p.M = g.M; p.N = g.N;
    p.kb_total = (int)((g.K + BK - 1) / BK);
    p.m_tiles = (int)((g.M + BM * cg - 1) / (BM * cg));
    p.n_tiles = (int)((g.N + bn - 1) / bn);
    p.bias = (const __nv_bfloat16*)g.bias;
    p.b_early = g.b_early;
    p.timeout_flag = device_timeout_flag();
    const int64_t tiles = (int64_t)p.m_tiles * p.n_tiles, units_max = kNumSms / cg;
    // every unit (block or pair) gets the same number of tiles (+-1): units = tiles / ceil(tiles / units_max), rounded up
    const int64_t waves = (tiles + units_max - 1) / units_max;
    const unsigned blocks = (unsigned)((tiles + waves - 1) / waves) * (unsigned)cg;
    if (cg == 2) {
        if (bn == 256) return launch_p_major<256, 2>(g.b_mn_major, tA, tB, tC, p, blocks, stream);
        return launch_p_major<128, 2>(g.b_mn_major, tA, tB, tC, p, blocks, stream);
    }
    switch (bn) {
        case 256: return launch_p_major<256, 1>(g.b_mn_major, tA, tB, tC, p, blocks, stream);
        case 192: return launch_p_major<192, 1>(g.b_mn_major, tA, tB, tC, p, blocks, stream);
        case 128: return launch_p_major<128, 1>(g.b_mn_major, tA, tB, tC, p, blocks, stream);
        default:  return launch_p_major<64, 1>(g.b_mn_major, tA, tB, tC, p, blocks, stream);
    }
}

}  // namespace lrd
