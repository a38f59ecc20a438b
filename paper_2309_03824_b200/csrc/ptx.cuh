// Thin inline-PTX wrappers for sm_100a: mbarrier, TMA (bulk tensor copies), tcgen05 (tensor
// memory, MMA, commit, loads), cluster barriers and distributed shared memory.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"

namespace lrd {
namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t elect_one() {
    uint32_t pred = 0;
    asm volatile(
        "{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred;
}

// ---- mbarrier -----------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}

__device__ __forceinline__ uint32_t mbar_test_wait(uint32_t bar, uint32_t parity) {     // never suspends
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}

// Bounded wait.  Returns false when the barrier did not flip within the limit or another
// thread of the block has already given up; the caller then leaves its loop and the block
// tears down in order.
constexpr uint32_t kWaitSpinFast = 1u << 14;
constexpr uint32_t kWaitSpinLimit = 1u << 22;
struct AbortCtx {
    volatile int* flag;        // shared memory: set by the first thread of the block that gives up
    unsigned int* global_flag; // device memory: reported to the host
};
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const AbortCtx& ab) {
    for (uint32_t it = 0; it < kWaitSpinLimit; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (it >= kWaitSpinFast) {                       // a try suspends in hardware for a while by itself; back
            __nanosleep(64);                             // off only when the wait is clearly a long one
            if (*ab.flag) return false;
        }
    }
    *ab.flag = 1;
    if (ab.global_flag) atomicExch(ab.global_flag, 1u);
    return false;
}

// The same wait executed by a whole converged warp, with a warp-uniform result (the warp stays
// converged, so that an elect.sync region can follow).
__device__ __forceinline__ bool mbar_wait_uniform(uint32_t bar, uint32_t parity, const AbortCtx& ab) {
    const bool ok = mbar_wait(bar, parity, ab);
    return __all_sync(0xffffffffu, ok) != 0;
}

// The same for a barrier that was looked at before (`ready` = mbar_test_wait of this phase, issued ahead of other work so
// that the hundred clocks a look takes pass beside it): waits only where that look came too early.
__device__ __forceinline__ bool mbar_wait_peeked(uint32_t ready, uint32_t bar, uint32_t parity, const AbortCtx& ab) {
    return __any_sync(0xffffffffu, ready == 0) ? mbar_wait_uniform(bar, parity, ab) : true;
}

// Warp-wide wait for the long waits of the epilogue warps: lane 0 polls with a sleep between tries
// (hot polling by many threads competes with the producer and MMA threads for issue slots), then
// every lane observes the completed phase itself.  Warp-uniform result.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, const AbortCtx& ab) {
    bool ok = true;
    if ((threadIdx.x & 31) == 0) {
        ok = false;
        for (uint32_t it = 0; it < kWaitSpinLimit; ++it) {
            if (mbar_try_wait(bar, parity)) { ok = true; break; }
            if (it >= 256) {
                __nanosleep(64);
                if (*ab.flag) break;
            }
        }
        if (!ok && !*ab.flag) {
            *ab.flag = 1;
            if (ab.global_flag) atomicExch(ab.global_flag, 1u);
        }
    }
    ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    if (ok) {
        for (int i = 0; i < 64 && !mbar_try_wait(bar, parity); ++i) {}
    }
    return ok;
}

// Cluster-scope wait: acquires what other blocks of the cluster released (data they copied into this
// block's shared memory completes on the barrier itself).
__device__ __forceinline__ uint32_t mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, const AbortCtx& ab) {
    for (uint32_t it = 0; it < kWaitSpinLimit; ++it) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        if (it >= kWaitSpinFast) {
            __nanosleep(128);
            if (*ab.flag) return false;
        }
    }
    *ab.flag = 1;
    if (ab.global_flag) atomicExch(ab.global_flag, 1u);
    return false;
}

__device__ __forceinline__ bool mbar_wait_cluster_uniform(uint32_t bar, uint32_t parity, const AbortCtx& ab) {
    const bool ok = mbar_wait_cluster(bar, parity, ab);
    return __all_sync(0xffffffffu, ok) != 0;
}

// ---- proxies and fences ---------------------------------------------------------------------
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---- TMA ----------------------------------------------------------------------------------------
__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)m) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"((uint64_t)m), "r"(bar), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2,
                                            int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"((uint64_t)m), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// im2col mode: `pixels` window positions from (w, h, n) on (coordinates of the window's first tap), at tap offset (ow, oh)
__device__ __forceinline__ void tma_load_im2col(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c, int w, int h, int n,
                                                uint32_t ow, uint32_t oh) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2], {%7, %8};"
        ::"r"(dst), "l"((uint64_t)m), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n), "h"((uint16_t)ow), "h"((uint16_t)oh) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* m, uint32_t src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"((uint64_t)m), "r"(src), "r"(x), "r"(y) : "memory");
}
// adds the tile to what is there (bf16: the sum rounded once)
__device__ __forceinline__ void tma_add_2d(const CUtensorMap* m, uint32_t src, int x, int y) {
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"((uint64_t)m), "r"(src), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void tma_store_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

// ---- tensor memory ------------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {   // whole warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {     // whole warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// D[tmem] (+)= A[smem desc] * B[smem desc], bf16 inputs, fp32 accumulate; one thread issues.
__device__ __forceinline__ void mma_bf16_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrive on an mbarrier once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 32 lanes x 32 consecutive fp32 columns: thread i of the warp gets lane (base lane + i).
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}
// 32 lanes x 16 consecutive fp32 columns.
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---- descriptors ------------------------------------------------------------------------------
// Shared-memory matrix descriptor, 128-byte swizzle.  lbo / sbo in bytes.
//   K-major operand  (rows of 64 bf16 = 128 B, 8-row groups of 1024 B): lbo unused, sbo = 1024.
//   MN-major operand (64-wide column blocks, each [k rows x 128 B]): lbo = bytes between column
//   blocks, sbo = bytes between 8-k-row groups (1024).
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;   // descriptor version of this architecture
    d |= (uint64_t)2 << 61;   // 128-byte swizzle
    return d;
}
// General form: swizzle span `swb` in {128, 64, 32} bytes.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo, uint32_t swb) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)(swb == 128 ? 2 : (swb == 64 ? 4 : 6)) << 61;
    return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = n (multiple of 16, <= 256).
__host__ __device__ constexpr uint32_t idesc_bf16(int n, bool a_mn_major, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) | ((b_mn_major ? 1u : 0u) << 16) |
           ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}

// ---- programmatic dependent launch ----------------------------------------------------------------
// A kernel launched with the programmatic-serialization attribute may start while its predecessor in
// the stream is still running.  launch_dependents: this block no longer holds the next kernel back.
// wait: returns once the predecessor has completed and its memory operations are visible; before it global memory
// may only be touched by the rule at GemmArgs::a_early.  Both are no-ops in a kernel launched without the attribute.
__device__ __forceinline__ void griddep_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- clusters -------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// Arrival without release semantics: signals progress only (a release waits for this block's
// outstanding asynchronous copies, which can take microseconds right after a push).
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Bulk copy from this block's shared memory into a peer block's shared memory (same offsets are the
// caller's business); completion is counted in bytes on the peer's mbarrier.
__device__ __forceinline__ void dsmem_bulk_copy(uint32_t dst_local_addr, uint32_t src_addr, uint32_t bytes,
                                                uint32_t bar_local_addr, uint32_t peer_rank) {
    asm volatile(
        "{\n\t.reg .b32 rd, rb;\n\t"
        "mapa.shared::cluster.u32 rd, %0, %4;\n\t"
        "mapa.shared::cluster.u32 rb, %3, %4;\n\t"
        "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [rd], [%1], %2, [rb];\n\t}"
        ::"r"(dst_local_addr), "r"(src_addr), "r"(bytes), "r"(bar_local_addr), "r"(peer_rank) : "memory");
}
__device__ __forceinline__ void named_bar_sync(int id, int nthreads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
// Barrier over `nthreads` threads that also ANDs a predicate across them.
__device__ __forceinline__ bool named_bar_and(int id, int nthreads, bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %3, 0;\n\tbar.red.and.pred p, %1, %2, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r) : "r"(id), "r"(nthreads), "r"(pred ? 1u : 0u) : "memory");
    return r != 0;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// The bias of an epilogue warp's four 32-column pieces of a tile (columns col0 + 64 e + lane), fetched a tile ahead into
// registers and put into shared memory (`at` = the place of col0) when the tile's turn comes.  Warps that share columns write
// the same values to the same place and each reads behind its own write; two tiles' bias alternate, and a tile's is
// written once its accumulator is complete, by when every warp is done with the tile two before it.
__device__ __forceinline__ void bias_fetch(uint16_t (&b)[4], const __nv_bfloat16* bias, int64_t col0, int64_t n) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int64_t col = col0 + 64 * e + (threadIdx.x & 31);
        b[e] = bias && col < n ? __bfloat16_as_ushort(bias[col]) : (uint16_t)0;
    }
}
__device__ __forceinline__ void bias_put(uint16_t* at, const uint16_t (&b)[4], int pieces) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (e < pieces) at[64 * e + (threadIdx.x & 31)] = b[e];
    __syncwarp();
}
// The same with the bias kept as fp32: twice the shared memory, half the instructions per piece, which a block of one or two
// chunks waits for (chain forward, 700 tokens, 512 -> 512 at rank 128: 6.53 us with bf16, 6.44 with fp32, 6.26 without a bias).
__device__ __forceinline__ void bias_put(float* at, const uint16_t (&b)[4], int pieces) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (e < pieces) at[64 * e + (threadIdx.x & 31)] = __uint_as_float((uint32_t)b[e] << 16);
    __syncwarp();
}
__device__ __forceinline__ void bias_add(uint32_t* v, const float* at) {
    const float4* bp = reinterpret_cast<const float4*>(at);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float4 b4 = bp[e];
        v[4 * e] = __float_as_uint(__uint_as_float(v[4 * e]) + b4.x);
        v[4 * e + 1] = __float_as_uint(__uint_as_float(v[4 * e + 1]) + b4.y);
        v[4 * e + 2] = __float_as_uint(__uint_as_float(v[4 * e + 2]) + b4.z);
        v[4 * e + 3] = __float_as_uint(__uint_as_float(v[4 * e + 3]) + b4.w);
    }
}
// 32 accumulators += bias of their columns
__device__ __forceinline__ void bias_add(uint32_t* v, const uint16_t* at) {
    const uint4* bp = reinterpret_cast<const uint4*>(at);
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const uint4 b4 = bp[x];
        const uint32_t w[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int y = 0; y < 4; ++y) {
            v[8 * x + 2 * y] = __float_as_uint(__uint_as_float(v[8 * x + 2 * y]) + __uint_as_float(w[y] << 16));
            v[8 * x + 2 * y + 1] = __float_as_uint(__uint_as_float(v[8 * x + 2 * y + 1]) + __uint_as_float(w[y] & 0xFFFF0000u));
        }
    }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

// A warp's `n` (<= 8) rows of at most 64 bf16 columns out of shared memory -- lane l's two of row i at src(i) -- to rows of any
// alignment, `to` = this lane's place in the first; `left`: columns from there on that exist.  All loads stand before all stores.
template <typename Src> __device__ __forceinline__ void store_any_rows8(const Src& src, int n, __nv_bfloat16* to, int64_t ld, int left) {
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v[i]) : "r"(src(i)));
    if (left <= 0) return;
    if (left > 1 && (((uintptr_t)to | (uintptr_t)(2 * ld)) & 3u) == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i, to += ld)
            if (i < n) *reinterpret_cast<uint32_t*>(to) = v[i];
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i, to += ld) {
            if (i >= n) continue;
            to[0] = __ushort_as_bfloat16((unsigned short)v[i]);
            if (left > 1) to[1] = __ushort_as_bfloat16((unsigned short)(v[i] >> 16));
        }
    }
}
// A slice of a chain's T buffer (columns [col0, col0 + n), atoms of [128 rows x taw columns], swizzled) to `rows` rows of a matrix
// that TMA cannot address, from buffer row `row0` (a multiple of 8) on, whole groups of eight rows readable.
__device__ __forceinline__ void store_slice_rows(uint32_t t_base, int taw, int col0, int n, int row0, int rows, __nv_bfloat16* dst, int64_t ld, int cols) {
    const uint32_t t_sw = 2u * (uint32_t)taw;
    for (int c = 2 * (int)(threadIdx.x & 31); c < n; c += 64) {
        const uint32_t gc = (uint32_t)(col0 + c), in = gc & ((uint32_t)taw - 1u), at = t_base + (gc / (uint32_t)taw) * 128u * t_sw + (in & 7u) * 2u;
        for (int r = 0; r < rows; r += 8)
            store_any_rows8([&](int i) { const uint32_t row = (uint32_t)(row0 + r + i); return at + row * t_sw + (((in / 8u) ^ ((row * t_sw >> 7) & (t_sw / 16u - 1u))) << 4); },
                            rows - r, dst + (int64_t)r * ld + gc, ld, cols - (int)gc);
    }
}

// One warp's 32 rows x 64 columns of bf16 out of shared memory (rows of 128 bytes, 16-byte groups swizzled by the row) to rows of
// `dst` (ld = cols of them, a multiple of 8): lane r's `row` is where row r goes, -1: nowhere.  Eight lanes share a row, so that an
// instruction writes four whole lines; stored straight from the registers, a lane a row, it touches 32.
__device__ __forceinline__ void store_rows64(uint32_t src, __nv_bfloat16* dst, int row, int col0, int cols) {
    const int lane = threadIdx.x & 31, col = col0 + 8 * (lane & 7);
    uint4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t r = 4u * i + ((uint32_t)lane >> 3);
        asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v[i].x), "=r"(v[i].y), "=r"(v[i].z), "=r"(v[i].w) : "r"(src + r * 128u + ((((uint32_t)lane & 7u) ^ (r & 7u)) << 4)));
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int to = __shfl_sync(0xffffffffu, row, 4 * i + (lane >> 3));
        if (to >= 0 && col < cols) *reinterpret_cast<uint4*>(dst + (int64_t)to * cols + col) = v[i];
    }
}
// 64 accumulators of this lane's row -> bf16, into the warp's rows of such a buffer
__device__ __forceinline__ void put_row64(uint32_t dst, const uint32_t (&v)[64]) {
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (uint32_t g = 0; g < 8; ++g)
        st_shared_v4(dst + lane * 128u + ((g ^ (lane & 7u)) << 4), pack_bf16(__uint_as_float(v[8 * g]), __uint_as_float(v[8 * g + 1])),
                     pack_bf16(__uint_as_float(v[8 * g + 2]), __uint_as_float(v[8 * g + 3])), pack_bf16(__uint_as_float(v[8 * g + 4]), __uint_as_float(v[8 * g + 5])),
                     pack_bf16(__uint_as_float(v[8 * g + 6]), __uint_as_float(v[8 * g + 7])));
}

// two bf16 sums, each fp32 and rounded once
__device__ __forceinline__ uint32_t add_bf16x2(uint32_t a, uint32_t b) {
    return pack_bf16(__uint_as_float(a << 16) + __uint_as_float(b << 16), __uint_as_float(a & 0xFFFF0000u) + __uint_as_float(b & 0xFFFF0000u));
}
__device__ __forceinline__ void add_into_bf16(__nv_bfloat16* dst, float x) {
    *dst = __float2bfloat16_rn(__bfloat162float(*dst) + __bfloat162float(__float2bfloat16_rn(x)));
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

}  // namespace ptx
}  // namespace lrd
