// Tensor-core k x k core convolution of the Tucker-2 layer (k = 1, 3, 5, 7; stride 1 or 2; zero pad (k - 1) / 2; NHWC,
// bf16) as an implicit GEMM on sm_100a.  No im2col buffer exists anywhere: the A operand of a filter tap is fetched by
// the TMA unit in im2col mode -- 128 consecutive output pixels (rows and images follow one another, so no tile has an
// unused row but the last) read at the tap's offset and the layer's stride, zeros outside the image = the padding.
//
//   conv_kernel<false>: forward        out[p][o] = sum_{tap,i} in[p stride + tap - pad][i] G[o][tap][i]
//   conv_kernel<true> : data gradient  din[q][i] = sum over (p, tap) with p stride + tap - pad = q, and o, of
//                       dout[p][o] G[o][tap][i].  With stride 2 the input pixels fall into four classes by the parity
//                       of their row and column; a class meets every second tap in each direction and is a stride-1
//                       convolution of dout with those taps (for k = 3: 4, 2, 2 and 1 of them).  A class has its own
//                       tensor map and its own tiles, those with the most taps first.
//   conv_kernel<.., true> (fused): the 1x1 product that follows the core runs in the same kernel.  The
//                       tile of the core's result is rounded to bf16 into shared memory (K-major,
//                       128-byte swizzle; written to memory only if the caller needs it), the ring,
//                       dead by then, receives the 1x1 factor Q[N2 x n1], and a second set of MMAs forms
//                       out2[p][:] = core[p][:] Q^T (+ bias) in the same tensor-memory columns:
//                       forward  Y = conv(Z1, G) Bm^T + b,  backward  dX = conv^T(dZ2, G) A^T.
// The filter gradient is a product over all pixels and runs on the weight-gradient kernel (tc_gemm.cu), whose second
// operand can be fetched in im2col mode too.
//
// A block takes at most half of an SM's shared and tensor memory where the grid has more blocks than the GPU has SMs,
// so that two blocks share an SM and one's set-up, first loads and epilogue run beside the other's MMAs.
// Warp roles as in the matrix-product kernel: TMA producer, MMA issuer (both issue under elect.sync from a converged
// warp), 8 epilogue warps: what a block does after its MMAs is latency of tensor-memory loads and stores, and more warps have
// more of both in flight.  A stride-2 step, 64 x 28 x 28, 256 -> 256 at rank 96: 65.6 us with four warps, 61.3 with eight and whole
// sectors per store; beside each other, sectors / whole lines out of shared memory 62.0 / 60.2 (replayed 56.6 / 54.7).
#include <algorithm>

#include "common.cuh"
#include "conv.cuh"
#include "ptx.cuh"
#include "tc.cuh"
#include "tma.cuh"

namespace lrd {
namespace {

using namespace ptx;

constexpr int kThreads = 320;                        // TMA producer, MMA issuer, 8 x epilogue
constexpr int kMaxStages = 8;
constexpr uint32_t kTile = 128 * 128;               // the A tile of a stage: 128 pixels x 64 channels of bf16
constexpr uint32_t kSmemFull = 222 * 1024, kSmemHalf = 110 * 1024;      // dynamic shared memory of one block per SM / two
constexpr int kMaxClasses = 4;

// The output pixels of one class: rows ph, ph + step, ... and columns pw, pw + step, ... of the output image, Hc x Wc
// of them per image.  They meet the taps (kh0 + a step, kw0 + b step), a < nkh, b < nkw; window position
// (h', w') starts at input row low_h + h' in_step, and tap (a, b) looks a (or, seen from the other side, nkh - 1 - a) further.
struct ConvClass {
    int pixels, tile0;            // pixels over all images; first tile of the class
    int Hc, Wc, ph, pw;
    int kh0, kw0, nkh, nkw, low_h, low_w;
};

struct ConvMaps {
    CUtensorMap img[kMaxClasses], g, q;
};

struct ConvParams {
    int H, W;                     // output image
    int step;                     // distance between the output pixels of a class (1, or 2 for a strided data gradient)
    int in_step;                  // distance between window positions in the input image (the stride in the forward pass, else 1)
    int k;
    int ka, nkc;                  // channels of the A-side image (reduction per tap) and 64-channel blocks of them
    int n_total;                  // output channels of this product (columns of out)
    int g_ci;                     // Ci of G[o][tap][i] (its row length is k * k * g_ci)
    int bn, stages;               // columns per block; ring stages of (16 KB + bn * 128 B)
    int tmem_cols;
    int n_cls;
    ConvClass cls[kMaxClasses];
    __nv_bfloat16* out;           // [pixels][n_total]; fused: nullable (the core's result is then never written to memory)
    unsigned int* timeout_flag;
    // fused 1x1 product
    int n2;                       // columns of out2 (<= 256)
    __nv_bfloat16* out2;          // [pixels][n2]
    const __nv_bfloat16* bias2;   // [n2] or nullptr
};

// grid: (tiles of all classes, column tiles of bn); fused: one column tile
template <bool DGRAD, bool FUSE>
__global__ void __launch_bounds__(kThreads, 2)
conv_kernel(const __grid_constant__ ConvMaps maps, const ConvParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], acc_bar, q_full, t_ready, out_full;
    __shared__ __align__(16) float bias_s[FUSE ? 256 : 1];
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_flag;
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const AbortCtx ab{&abort_flag, p.timeout_flag};
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x / 32, 0), lane = threadIdx.x % 32;
    int ci = 0;
    while (ci + 1 < p.n_cls && (int)blockIdx.x >= p.cls[ci + 1].tile0) ++ci;
    const ConvClass cl = p.cls[ci];
    const int m0 = ((int)blockIdx.x - cl.tile0) * 128;      // first pixel of the tile within the class
    const int n0 = FUSE ? 0 : (int)blockIdx.y * p.bn;
    const int iters = cl.nkh * cl.nkw * p.nkc;
    const uint32_t stage_bytes = kTile + (uint32_t)p.bn * 128u;

    if (threadIdx.x == 0) {
        abort_flag = 0;
        prefetch_tmap(&maps.img[ci]);
        prefetch_tmap(&maps.g);
        for (int s = 0; s < p.stages; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1);
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        mbar_init(smem_u32(&acc_bar), 1);
        mbar_init(smem_u32(&q_full), 1);
        mbar_init(smem_u32(&t_ready), 8);
        mbar_init(smem_u32(&out_full), 1);
        if (FUSE) prefetch_tmap(&maps.q);
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_base_slot), (uint32_t)p.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = tmem_base_slot;
    // set-up above touched only this block's own shared and tensor memory: under programmatic dependent launch it
    // overlaps the tail of the previous kernel in the stream; global memory is first touched below this line
    griddep_wait();
    griddep_launch_dependents();       // (in this order: see GemmArgs::a_early)
    // fused: once the core's MMAs are done the ring is dead; it then holds [T: one atom of 128 rows x 64 columns per 64
    // columns of the core's result | Q: one [n2 rows x 64 k] tile per 64 columns of the core's result]
    const int nq = (p.n_total + 63) / 64;
    const uint32_t q_tile = (uint32_t)p.n2 * 128u;
    const uint32_t t_base = smem_base, q_base = smem_base + (uint32_t)nq * kTile;

    if (warp == 0) {
        // TMA producer: the whole warp runs the loop, one elected lane issues
        const int w0 = cl.low_w + (m0 % cl.Wc) * p.in_step, h0 = cl.low_h + ((m0 / cl.Wc) % cl.Hc) * p.in_step;
        const int img = m0 / (cl.Wc * cl.Hc);
        int s = 0;
        uint32_t ph = 1;
        int a = 0, b = 0, cb = 0;                            // tap row, tap column, channel block
        for (int it = 0; it < iters; ++it) {
            if (!mbar_wait_uniform(smem_u32(&empty_bar[s]), ph, ab)) break;
            const uint32_t fb = smem_u32(&full_bar[s]);
            const uint32_t a_dst = smem_base + s * stage_bytes, b_dst = a_dst + kTile;
            const int g_col = ((cl.kh0 + a * p.step) * p.k + cl.kw0 + b * p.step) * p.g_ci;      // first column of this tap in G
            if (elect_one()) {
                mbar_expect_tx(fb, stage_bytes);
                tma_load_im2col(a_dst, &maps.img[ci], fb, cb * 64, w0, h0, img, (uint32_t)(DGRAD ? cl.nkw - 1 - b : b),
                                (uint32_t)(DGRAD ? cl.nkh - 1 - a : a));
                if (DGRAD) {           // B[n = i][k = o] = G[o][tap][i]: MN-major, rows o of this block, 64 columns of i per box
                    for (int j = 0; j < p.bn / 64; ++j) tma_load_2d(b_dst + j * 8192, &maps.g, fb, g_col + n0 + 64 * j, cb * 64);
                } else {               // B[n = o][k = i] = G[o][tap][i]: K-major, bn rows of o
                    tma_load_2d(b_dst, &maps.g, fb, g_col + cb * 64, n0);
                }
            }
            __syncwarp();
            if (++s == p.stages) { s = 0; ph ^= 1; }
            if (++cb == p.nkc) { cb = 0; if (++b == cl.nkw) { b = 0; ++a; } }
        }
        if (FUSE) {                                          // the 1x1 factor, into the dead ring (columns past n1: zeros)
            if (mbar_wait_uniform(smem_u32(&acc_bar), 0, ab)) {
                if (elect_one()) {
                    mbar_expect_tx(smem_u32(&q_full), (uint32_t)nq * q_tile);
                    for (int kb = 0; kb < nq; ++kb) tma_load_2d(q_base + kb * q_tile, &maps.q, smem_u32(&q_full), kb * 64, 0);
                }
                __syncwarp();
            }
        }
    } else if (warp == 1) {
        // MMA issuer: converged warp, elect.sync around the issue
        const uint32_t idesc = idesc_bf16(min(p.bn, (p.n_total - n0 + 15) / 16 * 16), false, DGRAD);
        int s = 0, cb = 0;
        uint32_t ph = 0;
        bool ok = true;
        uint32_t ready = mbar_test_wait(smem_u32(&full_bar[0]), 0);
        for (int it = 0; it < iters; ++it) {
            ok = mbar_wait_peeked(ready, smem_u32(&full_bar[s]), ph, ab);
            if (!ok) break;
            tc_fence_after();
            const uint32_t a_src = smem_base + s * stage_bytes, b_src = a_src + kTile, eb = smem_u32(&empty_bar[s]);
            if (++s == p.stages) { s = 0; ph ^= 1; }
            ready = mbar_test_wait(smem_u32(&full_bar[s]), ph);              // (after the last stage: not acted upon)
            const int nks = min(4, (p.ka - cb * 64 + 15) / 16);              // 16-channel steps past ka hold zeros: not issued
            if (elect_one()) {
                const uint64_t ad0 = smem_desc_sw128(a_src, 0, 1024);
                const uint64_t bd0 = DGRAD ? smem_desc_sw128(b_src, 8192, 1024) : smem_desc_sw128(b_src, 0, 1024);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)                               // the k-step moves the start address only
                    if (kk < nks) mma_bf16_ss(tmem_base, ad0 + 2u * kk, bd0 + (DGRAD ? 128u : 2u) * kk, idesc, (it > 0 || kk > 0) ? 1u : 0u);
                mma_commit(eb);
            }
            __syncwarp();
            if (++cb == p.nkc) cb = 0;
        }
        if (ok && elect_one()) mma_commit(smem_u32(&acc_bar));
        __syncwarp();
        if (FUSE) {                                          // out2 tile = T Q^T, reduction over the n_total columns of T
            // (t_ready also says that the core's accumulator, which these MMAs overwrite, has been read out)
            if (ok) ok = mbar_wait_uniform(smem_u32(&t_ready), 0, ab);
            if (ok) ok = mbar_wait_uniform(smem_u32(&q_full), 0, ab);
            if (ok) {
                tc_fence_after();
                const uint32_t idesc2 = idesc_bf16((p.n2 + 15) / 16 * 16, false, false);
                if (elect_one()) {
                    for (int ks = 0; ks * 16 < p.n_total; ++ks) {
                        const uint64_t ad = smem_desc_sw128(t_base + (ks / 4) * kTile + (ks % 4) * 32, 0, 1024);
                        const uint64_t bd = smem_desc_sw128(q_base + (ks / 4) * q_tile + (ks % 4) * 32, 0, 1024);
                        mma_bf16_ss(tmem_base, ad, bd, idesc2, ks > 0 ? 1u : 0u);
                    }
                    mma_commit(smem_u32(&out_full));
                }
                __syncwarp();
            }
        }
    } else {
        const int q = warp % 4, hw = (warp - 2) / 4;             // two warps share a quarter of the rows: alternate 64-column blocks
        const int m = m0 + q * 32 + lane;
        int pix = m < cl.pixels ? m : -1;                        // this lane's pixel of the output image(s); -1: none
        if (p.step > 1 && pix >= 0) {
            const int w = m % cl.Wc, h = (m / cl.Wc) % cl.Hc, im = m / (cl.Wc * cl.Hc);
            pix = (im * p.H + cl.ph + h * p.step) * p.W + cl.pw + w * p.step;
        }
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        if (FUSE)
            for (int n = threadIdx.x - 64; n < 256; n += 256) bias_s[n] = p.bias2 && n < p.n2 ? __bfloat162float(p.bias2[n]) : 0.f;
        const bool ready = mbar_wait_uniform(smem_u32(&acc_bar), 0, ab);
        tc_fence_after();
        // Blocks of 64 columns per warp, through shared memory: the T tile of the second product (rows past the tile hold garbage that
        // only reaches output rows nobody stores), or a slab of the warp in the dead ring; out of it to memory in whole lines.
        const uint32_t slab = smem_base + (uint32_t)(warp - 2) * 4096u;
        if (ready) {
#pragma unroll 1
            for (int c = 64 * hw; c < p.bn && n0 + c < p.n_total; c += 128) {
                uint32_t v[64];
                if (iters > 0) {
                    tmem_ld_32x32(lane_addr + c, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
                    tmem_ld_32x32(lane_addr + c + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
                    tmem_ld_wait();
                } else {                                         // a class that meets no tap (k = 1, stride 2)
#pragma unroll
                    for (int e = 0; e < 64; ++e) v[e] = 0u;
                }
                if (FUSE) {
                    put_row64(t_base + (uint32_t)(c / 64) * kTile + (uint32_t)q * 4096u, v);
                } else {
                    put_row64(slab, v);
                    __syncwarp();
                    store_rows64(slab, p.out, pix, n0 + c, p.n_total);
                    __syncwarp();
                }
            }
        }
        if (FUSE) {
            fence_proxy_async_smem();                        // T was written by ordinary stores, the MMA reads it through the async proxy
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&t_ready));
            if (ready && p.out)                              // the core's result, where it is wanted, while the second product runs
#pragma unroll 1
                for (int c = 64 * hw; c < p.n_total; c += 128) store_rows64(t_base + (uint32_t)(c / 64) * kTile + (uint32_t)q * 4096u, p.out, pix, c, p.n_total);
            const bool done = ready && mbar_wait_uniform(smem_u32(&out_full), 0, ab);
            tc_fence_after();
            named_bar_sync(2, 256);                          // (the bias is in shared memory, and every warp is done with T)
            if (done) {
#pragma unroll 1
                for (int col0 = 64 * hw; col0 < p.n2; col0 += 128) {
                    uint32_t v[64];
                    tmem_ld_32x32(lane_addr + col0, *reinterpret_cast<uint32_t(*)[32]>(&v[0]));
                    if (col0 + 32 < p.n2) tmem_ld_32x32(lane_addr + col0 + 32, *reinterpret_cast<uint32_t(*)[32]>(&v[32]));
                    tmem_ld_wait();
                    if (p.bias2) {
                        bias_add(&v[0], &bias_s[col0]);
                        bias_add(&v[32], &bias_s[col0 + 32]);
                    }
                    put_row64(slab, v);
                    __syncwarp();
                    store_rows64(slab, p.out2, pix, col0, p.n2);
                    __syncwarp();
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (abort_flag)
            for (int i = 0; i < 256; ++i) __nanosleep(1000);
        tc_fence_after();
        tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
}

inline bool a16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

int next_pow2(int x) {
    int n = 32;
    while (n < x) n *= 2;
    return n;
}

// Classes, tiles and tensor maps of one product.  dgrad = false: the A side is the input image (ci channels), the output
// pixels are those of the Ho x Wo grid; dgrad = true: the A side is the output gradient (co channels on the Ho x Wo
// grid), the output pixels those of the H x W grid.
bool setup(bool dgrad, const void* img, int64_t B, const ConvGeom& g, int64_t ci, int64_t co, ConvMaps* maps, ConvParams* p) {
    const int64_t ka = dgrad ? co : ci;
    p->k = g.k;
    p->ka = (int)ka;
    p->nkc = (int)((ka + 63) / 64);
    p->n_total = (int)(dgrad ? ci : co);
    p->g_ci = (int)ci;
    p->H = dgrad ? g.H : g.Ho;
    p->W = dgrad ? g.W : g.Wo;
    p->step = dgrad ? g.stride : 1;
    p->in_step = dgrad ? 1 : g.stride;
    const int in_h = dgrad ? g.Ho : g.H, in_w = dgrad ? g.Wo : g.W;
    int n = 0;
    for (int ph = 0; ph < p->step; ++ph)
        for (int pw = 0; pw < p->step; ++pw) {
            ConvClass c{};
            c.ph = ph; c.pw = pw;
            c.Hc = (p->H - ph + p->step - 1) / p->step;
            c.Wc = (p->W - pw + p->step - 1) / p->step;
            if (c.Hc < 1 || c.Wc < 1) continue;
            c.pixels = (int)(B * c.Hc * c.Wc);
            // taps kh0, kh0 + step, ...: those with (ph + pad - kh) divisible by the step (the forward pass meets all)
            c.kh0 = (ph + g.pad) % p->step;
            c.kw0 = (pw + g.pad) % p->step;
            c.nkh = c.kh0 < g.k ? (g.k - 1 - c.kh0) / p->step + 1 : 0;
            c.nkw = c.kw0 < g.k ? (g.k - 1 - c.kw0) / p->step + 1 : 0;
            if (c.nkh < 1 || c.nkw < 1) c.nkh = c.nkw = 0;
            // first input row / column a window position looks at
            c.low_h = dgrad ? (ph + g.pad - c.kh0) / p->step - (c.nkh - 1) : -g.pad;
            c.low_w = dgrad ? (pw + g.pad - c.kw0) / p->step - (c.nkw - 1) : -g.pad;
            p->cls[n++] = c;
        }
    p->n_cls = n;
    std::stable_sort(p->cls, p->cls + n, [](const ConvClass& a, const ConvClass& b) { return a.nkh * a.nkw > b.nkh * b.nkw; });
    int tiles = 0;
    for (int i = 0; i < n; ++i) {
        ConvClass& c = p->cls[i];
        c.tile0 = tiles;
        tiles += (c.pixels + 127) / 128;
        const bool taps = c.nkh > 0;                     // (a class without taps loads nothing; its map is never used)
        if (!make_tmap_im2col_bf16(&maps->img[i], img, (uint64_t)B, (uint64_t)in_h, (uint64_t)in_w, (uint64_t)ka, taps ? c.low_h : 0, taps ? c.low_w : 0,
                                   taps ? c.Hc : in_h, taps ? c.Wc : in_w, p->in_step, 128))
            return false;
    }
    for (int i = n; i < kMaxClasses; ++i) { p->cls[i] = p->cls[0]; maps->img[i] = maps->img[0]; }
    return true;
}

int total_tiles(const ConvParams& p) {
    const ConvClass& c = p.cls[p.n_cls - 1];
    return c.tile0 + (c.pixels + 127) / 128;
}

// Launch with the programmatic-serialization attribute: the kernel waits (griddepcontrol.wait) before it
// touches global memory, so its set-up may overlap the previous kernel's tail.
template <bool DGRAD, bool FUSE>
lrd_status_t launch_conv(const ConvMaps& maps, ConvParams& p, uint32_t fuse_bytes, cudaStream_t s) {
    auto kern = conv_kernel<DGRAD, FUSE>;
    static bool configured_on[kMaxDevices] = {};
    bool& configured = configured_on[device_slot()];
    if (!configured) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemFull) != cudaSuccess) return LRD_ERR_CUDA;
        configured = true;
    }
    const int tiles = total_tiles(p), n_tiles = (p.n_total + p.bn - 1) / p.bn;
    const uint32_t stage = kTile + (uint32_t)p.bn * 128u;
    const bool half = tiles * n_tiles > kNumSms && fuse_bytes + 1024u <= kSmemHalf && 2u * stage + 1024u <= kSmemHalf;
    p.stages = (int)std::min<uint32_t>(kMaxStages, ((half ? kSmemHalf : kSmemFull) - 1024u) / stage);
    p.tmem_cols = next_pow2(std::max(p.bn, FUSE ? p.n2 : 0));
    p.timeout_flag = device_timeout_flag();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles, (unsigned)n_tiles, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = 1024u + std::max((uint32_t)p.stages * stage, fuse_bytes);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (!cuda_ok(cudaLaunchKernelEx(&cfg, kern, maps, p), "cudaLaunchKernelEx(conv)")) return LRD_ERR_CUDA;
    count_launch();
    return LRD_OK;
}

// Columns per block of the unfused product: a stage costs its MMAs (2 bn clocks), its loads (about 80 B/clk into one SM)
// or the issue loop (some 500 clocks), whichever is longest, and a block some 5000 clocks beside its stages; the SM with
// the most blocks sets the pace.
int pick_bn(int64_t tiles, int64_t n_total, int64_t iters) {
    const int cands[4] = {256, 192, 128, 64};
    int best = 128;
    double best_cost = 1e300;
    for (int bn : cands) {
        if (bn > 64 && bn >= n_total + 64) continue;
        const int64_t blocks = tiles * ((n_total + bn - 1) / bn);
        const double stage = std::max({500.0, 2.0 * bn, (double)(kTile + bn * 128) / 80.0});
        const double cost = (double)((blocks + kNumSms - 1) / kNumSms) * ((double)iters * stage + 5000.0);
        if (cost < best_cost) { best_cost = cost; best = bn; }
    }
    return best;
}

bool geometry_ok(int64_t B, const ConvGeom& g, int64_t ci, int64_t co) {
    if (B < 1 || ci < 8 || co < 8 || ci % 8 || co % 8 || ci > (1 << 20) || co > (1 << 20)) return false;
    return B * g.H * g.W < ((int64_t)1 << 30);           // pixel indices are 32-bit
}

}  // namespace

bool tc_conv_eligible(int64_t B, const ConvGeom& g, int64_t ci, int64_t co, lrd_dtype_t dt, const void* p0, const void* p1, const void* p2) {
    return dt == LRD_BF16 && a16(p0) && a16(p1) && a16(p2) && geometry_ok(B, g, ci, co);
}

// forward (dgrad = false: img = in [..][ci], out [..][co]) or data gradient (dgrad = true: img = dout [..][co], out = din [..][ci])
lrd_status_t tc_conv(bool dgrad, const void* img, const void* G, void* out, int64_t B, const ConvGeom& g, int64_t ci, int64_t co,
                     cudaStream_t s) {
    if (!geometry_ok(B, g, ci, co)) return LRD_ERR_UNSUPPORTED;
    ConvMaps maps;
    ConvParams p{};
    if (!setup(dgrad, img, B, g, ci, co, &maps, &p)) return LRD_ERR_CUDA;
    const int64_t taps = (int64_t)g.k * g.k;
    p.bn = pick_bn(total_tiles(p), p.n_total, (int64_t)p.nkc * taps / (p.step * p.step));
    if (!make_tmap_2d_bf16(&maps.g, G, (uint64_t)co, (uint64_t)(taps * ci), (uint64_t)(taps * ci), dgrad ? 64u : (uint32_t)p.bn, 64)) return LRD_ERR_CUDA;
    maps.q = maps.g;
    p.out = (__nv_bfloat16*)out;
    return dgrad ? launch_conv<true, false>(maps, p, 0, s) : launch_conv<false, false>(maps, p, 0, s);
}

int64_t tc_conv_blocks(bool dgrad, bool fused, int64_t B, const ConvGeom& g, int64_t ci, int64_t co) {
    const int64_t tiles = (B * (dgrad ? (int64_t)g.H * g.W : (int64_t)g.Ho * g.Wo) + 127) / 128, n = dgrad ? ci : co, ka = dgrad ? co : ci;
    if (fused) return tiles;
    const int bn = pick_bn(tiles, n, (ka + 63) / 64 * g.k * g.k / (dgrad ? g.stride * g.stride : 1));
    return tiles * ((n + bn - 1) / bn);
}

bool tc_conv_chain_eligible(bool dgrad, int64_t B, const ConvGeom& g, int64_t ci, int64_t co, int64_t n2, lrd_dtype_t dt,
                            const void* img, const void* G, const void* Q, const void* out2, const void* core_out) {
    const int64_t n1 = dgrad ? ci : co;                  // channels of the core's result = reduction of the 1x1 product
    if (!tc_conv_eligible(B, g, ci, co, dt, img, G, Q)) return false;
    if (n1 > 256 || n1 % 16 || n2 < 8 || n2 > 256 || n2 % 8) return false;
    return a16(out2) && (!core_out || a16(core_out));
}

// The core followed by the 1x1 product out2[p][:] = core[p][:] Q^T (+ bias2) in one launch.  Q is [n2 x n1] with n1
// contiguous; core_out (nullable) receives the core's bf16 result when the caller needs it later.
lrd_status_t tc_conv_chain(bool dgrad, const void* img, const void* G, const void* Q, const void* bias2, void* out2, void* core_out,
                           int64_t B, const ConvGeom& g, int64_t ci, int64_t co, int64_t n2, cudaStream_t s) {
    if (!geometry_ok(B, g, ci, co)) return LRD_ERR_UNSUPPORTED;
    const int64_t n1 = dgrad ? ci : co, taps = (int64_t)g.k * g.k;
    ConvMaps maps;
    ConvParams p{};
    if (!setup(dgrad, img, B, g, ci, co, &maps, &p)) return LRD_ERR_CUDA;
    p.bn = (int)((n1 + 63) / 64 * 64);
    p.n2 = (int)n2;
    bool ok = make_tmap_2d_bf16(&maps.g, G, (uint64_t)co, (uint64_t)(taps * ci), (uint64_t)(taps * ci), dgrad ? 64u : (uint32_t)p.bn, 64);
    ok = ok && make_tmap_2d_bf16(&maps.q, Q, (uint64_t)n2, (uint64_t)n1, (uint64_t)n1, (uint32_t)n2, 64);
    if (!ok) return LRD_ERR_CUDA;
    p.out = (__nv_bfloat16*)core_out;
    p.out2 = (__nv_bfloat16*)out2;
    p.bias2 = (const __nv_bfloat16*)bias2;
    // (an MMA reads whole groups of 16 rows of Q: up to 8 rows past the last tile)
    const uint32_t fuse_bytes = (uint32_t)((n1 + 63) / 64) * (kTile + (uint32_t)n2 * 128u) + 1024u * (uint32_t)(n2 % 16 != 0);
    return dgrad ? launch_conv<true, true>(maps, p, fuse_bytes, s) : launch_conv<false, true>(maps, p, fuse_bytes, s);
}

}  // namespace lrd
