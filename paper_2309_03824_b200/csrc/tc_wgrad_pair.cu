// Weight gradients on pairs of SMs (sm_100a):  C[M x N] = A^T B, A[K x M] and B[K x N] both MN-major, the reduction over K
// tokens split over the pairs of a cluster; optionally the sums of A over k (the bias gradient: A = dY).
//
// A cluster of 2 S blocks owns one 256 x BN tile of C.  Blocks 2 p and 2 p + 1 are MMA pair p (tcgen05 cta_group::2): they
// take share p of the k-blocks, block h of the pair loads rows [128 h, 128 h + 128) of the tile's A and HALF of its B, and
// the even block issues 256-row MMAs.  Per k-block an SM then loads 16 KB + BN * 64 B for 128 x BN products where the
// single-block kernel (tc_gemm.cu) loads 16 KB + BN * 128 B, and its tensor pipe runs at N = 256.
// The partial tiles are reduced as in that kernel: every block sends each peer with the same rows the columns that peer
// owns (fp32, bulk DSMEM copies) and adds what it receives in rank order -- its own columns stay in tensor memory, so
// the staging takes 2 (S - 1) / S of a tile.  One launch, no scratch, bit-reproducible.
// Column sums: one more MMA per k-step, 16 columns wide, against a block of ones (any layout of ones is the same).
// What bounds it: the tensor pipe at BN = 256 (0.40 us per k-block of a pair, 1.55 PFLOP/s when all pairs run), shared memory's read
// rate at BN = 128 (0.26), and some 7 us of launch, first loads, exchange and stores.  4096 x 512 over 8192 tokens with the
// column sums: 33.4 us, 41.5 as two shares through scratch memory on tc_gemm.cu; 4096 x 1024 over 1024 tokens 11.8 from 16.2.
// Where tc_gemm.cu can give each tile a cluster of its own the smaller blocks are as fast or faster (3072 x 384 over 4096: 15
// against 20), so the dispatch compares estimates.  Two k-blocks per stage at BN = 256 and a second producer warp for B: no gain.
// Warp 0: TMA producer.  Warp 1: tensor memory, in the even block MMA issue.  Warps 2-9: reduction and stores.
// Every wait is bounded; a wait that runs out raises the device timeout flag and the cluster tears down in order.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "ptx_pair.cuh"
#include "tc.cuh"
#include "tma.cuh"

namespace lrd {
namespace {

using namespace ptx;

constexpr int BK = 64, kThreads = 320;
constexpr int kMaxPairs = 4;                          // portable cluster size
constexpr uint32_t kRingBytes = 192 * 1024, kOnesBytes = 2048;
constexpr uint32_t kSmemBytes = 1024 + kRingBytes + kOnesBytes;

// G: 64-deep k-blocks per stage (two for the narrow tile, see tc_gemm_persistent.cu)
template <int BN> struct Cfg {
    static constexpr int G = BN <= 128 ? 2 : 1;
    static constexpr uint32_t BOX = 8192u * G;                        // 64 G k rows x 64 columns
    static constexpr uint32_t A_BYTES = 2 * BOX, B_BYTES = BN / 128 * BOX, STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = kRingBytes / STAGE_BYTES;
    static constexpr uint32_t TMEM_COLS = BN <= 128 ? 256 : 512;      // tile + 16 columns of sums
};

struct WgradParams {
    int64_t M, N, ldc;
    int kb_total, kb_per_pair;
    __nv_bfloat16* C;
    __nv_bfloat16* colsum;        // [M] or nullptr
};
// NP independent products at most: their row tiles follow one another in gridDim.z.
template <int NP> struct WgradLaunch {
    unsigned int* timeout_flag;
    int pairs;
    int row0[NP];                 // first row tile of each (INT_MAX: none)
    WgradParams p[NP];
    CUtensorMap tA[NP], tB[NP];
};

// 16 columns of one row, rounded once (ADD: added to what C holds, see tc_gemm.cu)
template <bool ADD>
__device__ __forceinline__ void store16(const WgradParams& p, int64_t row, int64_t col, const float (&f)[16], bool sectors) {
    if (row >= p.M || col >= p.N) return;
    __nv_bfloat16* dst = p.C + row * p.ldc + col;
    uint32_t w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = pack_bf16(f[2 * e], f[2 * e + 1]);
    if (col + 16 <= p.N && sectors) {
        if (ADD) {
            const uint4 o0 = reinterpret_cast<const uint4*>(dst)[0], o1 = reinterpret_cast<const uint4*>(dst)[1];
            const uint32_t o[8] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) w[e] = add_bf16x2(w[e], o[e]);
        }
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
        return;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (col + 8 * h + 8 <= p.N) {
            if (ADD) {
                const uint4 o = *reinterpret_cast<const uint4*>(dst + 8 * h);
                w[4 * h] = add_bf16x2(w[4 * h], o.x); w[4 * h + 1] = add_bf16x2(w[4 * h + 1], o.y);
                w[4 * h + 2] = add_bf16x2(w[4 * h + 2], o.z); w[4 * h + 3] = add_bf16x2(w[4 * h + 3], o.w);
            }
            *reinterpret_cast<uint4*>(dst + 8 * h) = make_uint4(w[4 * h], w[4 * h + 1], w[4 * h + 2], w[4 * h + 3]);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (col + 8 * h + e < p.N) {
                    if (ADD) add_into_bf16(dst + 8 * h + e, f[8 * h + e]);
                    else dst[8 * h + e] = __float2bfloat16_rn(f[8 * h + e]);
                }
        }
    }
}

// grid: (2 pairs = one cluster, column tiles, row tiles of 256)
template <int BN, int NP, bool ADD>
__global__ void __launch_bounds__(kThreads, 1)
wgrad_pair_kernel(const __grid_constant__ WgradLaunch<NP> L) {
    int prod = 0;
#pragma unroll
    for (int i = 1; i < NP; ++i)
        if ((int)blockIdx.z >= L.row0[i]) prod = i;
    const CUtensorMap &tmA = L.tA[prod], &tmB = L.tB[prod];
    const WgradParams p = L.p[prod];
    if (NP > 1 && (int64_t)blockIdx.y * BN >= p.N) return;         // (the whole cluster: its blocks share y and z)
    using C = Cfg<BN>;
    constexpr int STAGES = C::STAGES, G = C::G;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[STAGES], empty_bar[STAGES], acc_bar, red_bar;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    const uint32_t ring_base = (smem_u32(smem_raw) + 1023u) & ~1023u, ones_base = ring_base + kRingBytes;
    const AbortCtx ab{&abort_flag, L.timeout_flag};
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    const uint32_t crank = cluster_ctarank();
    const int S = L.pairs, pr = (int)(crank >> 1), h = (int)(crank & 1u);
    const uint32_t lead_rank = crank & ~1u;
    const uint16_t pair_mask = (uint16_t)(3u << lead_rank);
    const int m0 = ((int)blockIdx.z - (NP > 1 ? L.row0[prod] : 0)) * 256 + h * 128, n0 = (int)blockIdx.y * BN;
    const int kb_begin = min(pr * p.kb_per_pair, p.kb_total), kb_end = min(kb_begin + p.kb_per_pair, p.kb_total);
    const bool sums = p.colsum != nullptr && blockIdx.y == 0;
    const uint32_t cs = (uint32_t)(BN / S), chunk_bytes = 128u * cs * 4u;       // columns this block owns; one slice of them
    // after the main loop: [S - 1 slices to send | S - 1 slices received | column sums to send | column sums received]
    const uint32_t send_base = ring_base, recv_base = ring_base + (uint32_t)(S - 1) * chunk_bytes, cs_send = ones_base, cs_recv = ones_base + 512u;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        mbar_init(smem_u32(&acc_bar), 1);
        mbar_init(smem_u32(&red_bar), 1);
        if (S > 1) mbar_expect_tx(smem_u32(&red_bar), (uint32_t)(S - 1) * (chunk_bytes + (sums && pr == 0 ? 512u : 0u)));
        fence_mbar_init();
    }
    if (threadIdx.x >= 64 && threadIdx.x < 64 + kOnesBytes / 16)
        st_shared_v4(ones_base + (threadIdx.x - 64) * 16u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
    fence_proxy_async_smem();
    if (warp == 1) {
        tmem_alloc_pair(smem_u32(&tmem_base_slot), C::TMEM_COLS);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive();              // every block's barriers (and ones) exist before a partner or a peer uses them
    cluster_wait();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    // set-up above touched only shared and tensor memory: it may overlap the tail of the previous kernel in the stream;
    // global memory is first touched below this line
    griddep_launch_dependents();       // (before the wait: nothing for an early launch to rely on, see GemmArgs::a_early)
    griddep_wait();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        int s = 0;
        uint32_t ph = 1;
        const int b0 = n0 + h * (BN / 2);
        for (int kb = kb_begin; kb < kb_end; kb += G) {      // (a k-block past this pair's share is loaded, not multiplied)
            if (!mbar_wait_uniform(smem_u32(&empty_bar[s]), ph, ab)) break;
            const uint32_t fb = map_to_cta(smem_u32(&full_bar[s]), lead_rank);   // the pair's loads complete on the even block's barrier
            const uint32_t dst = ring_base + (uint32_t)s * C::STAGE_BYTES;
            if (elect_one()) {
                if (h == 0) mbar_expect_tx(smem_u32(&full_bar[s]), 2u * C::STAGE_BYTES);
#pragma unroll
                for (int j = 0; j < 2; ++j) tma_load_2d_pair(dst + j * C::BOX, &tmA, fb, m0 + 64 * j, kb * BK);
#pragma unroll
                for (int j = 0; j < BN / 128; ++j) tma_load_2d_pair(dst + C::A_BYTES + j * C::BOX, &tmB, fb, b0 + 64 * j, kb * BK);
            }
            __syncwarp();
            if (++s == STAGES) { s = 0; ph ^= 1; }
        }
        cluster_arrive_relaxed(); cluster_wait(); cluster_arrive_relaxed();       // barriers 1 and 2, see the reduction
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (the even block)
        if (h == 0) {
            constexpr uint32_t idesc = idesc_bf16_pair(BN, true, true), idesc_sums = idesc_bf16_pair(16, true, true);
            const uint64_t a_desc0 = smem_desc_sw128(ring_base, C::BOX, 1024), b_desc0 = smem_desc_sw128(ring_base + C::A_BYTES, C::BOX, 1024);
            const uint64_t ones_desc = smem_desc_sw128(ones_base, 0, 1024);
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
                    for (int ks = 0; ks < 4 * G; ++ks) {
                        if (ks >= 4 && kb + 1 >= kb_end) break;
                        const uint32_t acc = ks > 0 ? 1u : (kb > kb_begin ? 1u : 0u);
                        mma_bf16_ss_pair(tmem_base, ad + ks * 128u, bd + ks * 128u, idesc, acc);
                        if (sums) mma_bf16_ss_pair(tmem_base + BN, ad + ks * 128u, ones_desc, idesc_sums, acc);
                    }
                    mma_commit_pair(eb, pair_mask);
                }
                __syncwarp();
            }
            if (ok && elect_one()) mma_commit_pair(smem_u32(&acc_bar), pair_mask);
            __syncwarp();
        }
        cluster_arrive_relaxed(); cluster_wait(); cluster_arrive_relaxed();
    } else {
        // ------------------------------------------------------------------ reduction and stores
        const int q = warp % 4, hw = (warp - 2) / 4;         // two warps share a quarter of the rows: alternate pieces of columns
        const int row = q * 32 + lane;
        const int64_t grow = (int64_t)m0 + row;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const bool has_work = kb_begin < kb_end;             // a pair past the end of the reduction contributes zeros
        const bool sectors = p.ldc % 16 == 0 && ((uintptr_t)p.C & 31u) == 0;
        const uint32_t ngrp = cs / 4u, rot = (uint32_t)row % ngrp;   // 16-byte groups of a row, rotated by the row: no two rows of a warp hit the same banks
        if (ADD && grow < p.M) {       // what this block's columns add to, on its way while the products are formed
            for (uint32_t c = (uint32_t)hw * 64u; c < cs; c += 128u)
                if ((int64_t)n0 + pr * cs + c < p.N) prefetch_l2(p.C + grow * p.ldc + n0 + pr * cs + c);
        }
        bool ok = mbar_wait_warp(smem_u32(&acc_bar), 0, ab);
        tc_fence_after();
        cluster_arrive_relaxed();      // barrier 1: this block's ring is dead (progress only)
        if (ok && S > 1) {
            // the peers' columns -> staging, [owner][row][cs]
            for (int piece = hw; piece < BN / 32; piece += 2) {
                const int owner = piece * 32 / (int)cs;
                if (owner == pr) continue;
                uint32_t v[32];
                if (has_work) {
                    tmem_ld_32x32(lane_addr + piece * 32, v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = 0u;
                }
                const uint32_t slot = (uint32_t)(owner < pr ? owner : owner - 1);
                const uint32_t dst_row = send_base + slot * chunk_bytes + (uint32_t)row * cs * 4u, g0 = ((uint32_t)piece * 32u - (uint32_t)owner * cs) / 4u;
#pragma unroll
                for (int g = 0; g < 8; ++g) {
                    uint32_t rg = g0 + g + rot;
                    if (rg >= ngrp) rg -= ngrp;
                    st_shared_v4(dst_row + rg * 16u, v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
                }
            }
        }
        float own_sum = 0.f;
        if (ok && sums && hw == 0) {
            uint32_t cv[16];
            if (has_work) {
                tmem_ld_32x16(lane_addr + BN, cv);
                tmem_ld_wait();
                own_sum = __uint_as_float(cv[0]);
            }
            if (pr != 0) asm volatile("st.shared.f32 [%0], %1;" ::"r"(cs_send + (uint32_t)row * 4u), "f"(own_sum) : "memory");
        }
        fence_proxy_async_smem();
        tc_fence_before();
        cluster_wait();                // barrier 1 complete: every peer's ring is dead, its receive slots may be written
        ok = named_bar_and(2, 256, ok);
        if (warp == 2 && S > 1) {
            if (ok && elect_one()) {
                for (int t = 1; t < S; ++t) {
                    const int peer = (pr + t) % S;
                    const uint32_t from = (uint32_t)(peer < pr ? peer : peer - 1), to = (uint32_t)(pr < peer ? pr : pr - 1);
                    dsmem_bulk_copy(recv_base + to * chunk_bytes, send_base + from * chunk_bytes, chunk_bytes, smem_u32(&red_bar), (uint32_t)(2 * peer + h));
                }
                if (sums && pr != 0) dsmem_bulk_copy(cs_recv + (uint32_t)(pr - 1) * 512u, cs_send, 512u, smem_u32(&red_bar), (uint32_t)h);
            }
            __syncwarp();
        }
        if (ok && S > 1) {
            bool got = false;
            if (lane == 0) got = mbar_wait_cluster(smem_u32(&red_bar), 0, ab);
            ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
            if (ok) { for (int i = 0; i < 64 && !mbar_try_wait_cluster(smem_u32(&red_bar), 0); ++i) {} }
        }
        cluster_arrive_relaxed();      // barrier 2: everything addressed to this block has landed (progress only)
        tc_fence_after();
        if (ok) {
            // this block's columns: the partials in rank order, its own out of tensor memory, rounded once
            for (uint32_t c0 = (uint32_t)hw * 32u; c0 < cs; c0 += 64u) {
                uint32_t own[32];
                if (has_work) {
                    tmem_ld_32x32(lane_addr + (uint32_t)pr * cs + c0, own);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int e = 0; e < 32; ++e) own[e] = 0u;
                }
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    float f[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) f[e] = 0.f;
#pragma unroll 1
                    for (int k = 0; k < S; ++k) {
                        if (k == pr) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) f[e] += __uint_as_float(own[16 * half + e]);
                            continue;
                        }
                        const uint32_t src = recv_base + (uint32_t)(k < pr ? k : k - 1) * chunk_bytes + (uint32_t)row * cs * 4u;
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            uint32_t rg = (c0 + 16u * half) / 4u + g + rot;
                            if (rg >= ngrp) rg -= ngrp;
                            float4 x;
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(src + rg * 16u));
                            f[4 * g] += x.x; f[4 * g + 1] += x.y; f[4 * g + 2] += x.z; f[4 * g + 3] += x.w;
                        }
                    }
                    store16<ADD>(p, grow, (int64_t)n0 + pr * cs + c0 + 16 * half, f, sectors);
                }
            }
            if (sums && hw == 0 && pr == 0 && grow < p.M) {
                float t = own_sum;
                for (int k = 1; k < S; ++k) {
                    float x;
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(cs_recv + (uint32_t)(k - 1) * 512u + (uint32_t)row * 4u));
                    t += x;
                }
                if (ADD) add_into_bf16(p.colsum + grow, t);
                else p.colsum[grow] = __float2bfloat16_rn(t);
            }
        }
        tc_fence_before();
    }
    // barrier 2: no block leaves (or frees tensor memory) while a peer may still read a slice out of its shared memory, or its
    // partner's MMAs and commits still reach it
    cluster_wait();
    __syncthreads();
    if (warp == 1) {
        if (abort_flag) {            // give copies and MMAs still in flight time to land before freeing
            for (int i = 0; i < 256; ++i) __nanosleep(1000);
        }
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
    }
}

bool set_attributes() {
    auto one = [](const void* f) { return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes) == cudaSuccess; };
    return one((const void*)wgrad_pair_kernel<256, 1, false>) && one((const void*)wgrad_pair_kernel<128, 1, false>) &&
           one((const void*)wgrad_pair_kernel<256, kMaxWgrads, false>) && one((const void*)wgrad_pair_kernel<256, 1, true>) &&
           one((const void*)wgrad_pair_kernel<128, 1, true>) && one((const void*)wgrad_pair_kernel<256, kMaxWgrads, true>);
}

// Clusters of n blocks that can be resident at once.
int max_active_clusters(int n) {
    static int cache_on[kMaxDevices][2 * kMaxPairs + 1] = {};
    int* cache = cache_on[device_slot()];
    if (cache[n] == 0) {
        int cnt = 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)n, 1, 1);
        cfg.blockDim = dim3(kThreads, 1, 1);
        cfg.dynamicSmemBytes = kSmemBytes;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)n;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (!set_attributes() || cudaOccupancyMaxActiveClusters(&cnt, wgrad_pair_kernel<256, 1, false>, &cfg) != cudaSuccess || cnt < 1) {
            cudaGetLastError();
            cnt = (kNumSms - 20) / n;
        }
        cache[n] = cnt;
    }
    return cache[n];
}

struct Plan { int bn, pairs; double us; };

// Estimated microseconds: 3 of launch and first loads, the k-blocks of a pair's share, 1.5 of stores, 2.5 of exchange (measured
// at 4096 x 512 over 8192 tokens: 256 wide one pair 54.9, two 33.3, 128 wide one pair 36.0); every further wave pays for its
// first loads too (4096 x 4096 over 2048 tokens, four waves: 73.0, as 192 wide tiles of single SMs 69.1).
Plan make_plan(const GemmArgs* g, int n) {
    Plan best{0, 0, 1e300};
    bool sums = false;
    int64_t kb = 0;
    for (int i = 0; i < n; ++i) {
        sums = sums || g[i].a_colsum;
        kb = std::max(kb, (g[i].K + BK - 1) / BK);
    }
    for (int bn : {256, 128}) {
        if (n > 1 && bn == 128) continue;                 // several products fill the narrow tiles' SMs better as single blocks
        int64_t tiles = 0;
        for (int i = 0; i < n; ++i) tiles += ((g[i].M + 255) / 256) * ((g[i].N + bn - 1) / bn);
        for (int S = kMaxPairs; S >= 1; S /= 2) {
            if ((g[0].max_cluster_split && 2 * S > g[0].max_cluster_split) || S > kb) continue;
            const int64_t room = max_active_clusters(2 * S), waves = (tiles + room - 1) / room;
            if (S > 1 && waves > 1) continue;
            const double per = (bn == 256 ? 0.40 : 0.25) + (sums ? 0.01 : 0.0);
            const double us = (double)waves * ((double)((kb + S - 1) / S) * per + (S > 1 ? 4.0 : 1.5)) + 3.0 * (double)waves;
            if (us < best.us) best = Plan{bn, S, us};
        }
    }
    return best;
}

}  // namespace

double tc_wgrad_pair_estimate(const GemmArgs* g, int n) {
    int64_t rows = 0;
    if (n > kMaxWgrads) return 1e300;
    for (int i = 0; i < n; ++i) {
        if (g[i].any_rows || !tc_gemm_eligible(g[i]) || !g[i].a_mn_major || !g[i].b_mn_major || g[i].bias || g[i].N > (int64_t)65535 * 128) return 1e300;
        rows += (g[i].M + 255) / 256;
    }
    return rows > 65535 ? 1e300 : make_plan(g, n).us;
}

template <int NP>
static lrd_status_t launch(const GemmArgs* g, int n, const Plan& pl, cudaStream_t stream) {
    const uint32_t box = BK * (uint32_t)(pl.bn == 256 ? Cfg<256>::G : Cfg<128>::G);
    WgradLaunch<NP> L{};
    unsigned ny = 0, nz = 0;
    for (int i = 0; i < NP; ++i) {
        L.row0[i] = i < n ? (int)nz : INT_MAX;
        if (i >= n) continue;
        if (!make_tmap_2d_bf16(&L.tA[i], g[i].A, (uint64_t)g[i].K, (uint64_t)g[i].M, (uint64_t)g[i].lda, box, 64) ||
            !make_tmap_2d_bf16(&L.tB[i], g[i].B, (uint64_t)g[i].K, (uint64_t)g[i].N, (uint64_t)g[i].ldb, box, 64))
            return LRD_ERR_CUDA;
        WgradParams& p = L.p[i];
        p.M = g[i].M; p.N = g[i].N; p.ldc = g[i].ldc;
        p.kb_total = (int)((g[i].K + BK - 1) / BK);
        p.kb_per_pair = (p.kb_total + pl.pairs - 1) / pl.pairs;
        p.C = (__nv_bfloat16*)g[i].C;
        p.colsum = (__nv_bfloat16*)g[i].a_colsum;
        ny = std::max(ny, (unsigned)((g[i].N + pl.bn - 1) / pl.bn));
        nz += (unsigned)((g[i].M + 255) / 256);
    }
    L.pairs = pl.pairs;
    L.timeout_flag = device_timeout_flag();
    static bool configured_on[kMaxDevices] = {};
    bool& configured = configured_on[device_slot()];
    if (!configured) {
        if (!set_attributes()) return LRD_ERR_CUDA;
        configured = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pl.pairs), ny, nz);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)(2 * pl.pairs);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the kernel waits (griddepcontrol.wait) before it touches global memory
    attr[1].val.programmaticStreamSerializationAllowed = g[0].in_turn ? 0 : 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    auto kern = g[0].add ? wgrad_pair_kernel<256, NP, true> : wgrad_pair_kernel<256, NP, false>;
    if constexpr (NP == 1)
        if (pl.bn == 128) kern = g[0].add ? wgrad_pair_kernel<128, 1, true> : wgrad_pair_kernel<128, 1, false>;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, L);
    if (!cuda_ok(e, "cudaLaunchKernelEx(weight gradient on pairs)")) return LRD_ERR_CUDA;
    count_launch();
    return LRD_OK;
}

lrd_status_t tc_wgrad_pair(const GemmArgs* g, int n, cudaStream_t stream) {
    if (tc_wgrad_pair_estimate(g, n) >= 1e300) return LRD_ERR_UNSUPPORTED;
    const WgradForm& form = tc_wgrad_form();
    const Plan pl = form.blocks == 2 ? Plan{form.columns, form.split, 0.0} : make_plan(g, n);
    if (n > 1 && pl.bn != 256) return LRD_ERR_UNSUPPORTED;
    return n == 1 ? launch<1>(g, n, pl, stream) : launch<kMaxWgrads>(g, n, pl, stream);
}

}  // namespace lrd
