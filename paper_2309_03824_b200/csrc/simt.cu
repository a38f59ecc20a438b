// General path: shared-memory tiled fp32-FMA matrix product for any shape, leading dimension and
// operand orientation (the column sums of its A operand a by-product where asked for).  Used for fp32 layers (which must not use
// reduced-precision tensor math) and for bf16 layers whose ranks or strides do not meet the
// 16-byte alignment the tensor-core path needs.
#include <cooperative_groups.h>

#include "common.cuh"
#include "conv.cuh"
#include "ptx.cuh"
#include "tc.cuh"

namespace cg = cooperative_groups;

namespace lrd {

__device__ unsigned int g_device_timeout = 0;

unsigned int* device_timeout_flag() {
    static unsigned int* ptr_on[kMaxDevices] = {};          // every device has its own copy of the symbol
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    void* p = nullptr;
    if (dev < 0 || dev >= kMaxDevices)                      // past the table: look it up every time
        return cudaGetSymbolAddress(&p, g_device_timeout) == cudaSuccess ? (unsigned int*)p : nullptr;
    if (!ptr_on[dev] && cudaGetSymbolAddress(&p, g_device_timeout) == cudaSuccess) ptr_on[dev] = (unsigned int*)p;
    return ptr_on[dev];
}

lrd_status_t read_and_clear_device_timeout(bool* raised) {
    unsigned int flag = 0;
    if (cudaMemcpyFromSymbol(&flag, g_device_timeout, sizeof(flag)) != cudaSuccess) return LRD_ERR_CUDA;
    *raised = flag != 0;
    if (flag) {
        const unsigned int zero = 0;
        if (cudaMemcpyToSymbol(g_device_timeout, &zero, sizeof(zero)) != cudaSuccess) return LRD_ERR_CUDA;
    }
    return LRD_OK;
}

namespace {

__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// Operand loaders: element (m, k) of A and (k, n) of B as fp32, asked for inside the problem only.  What depends on the
// row of A or the column of B alone (divisions by image sizes, mostly) is worked out once per thread and row: `row(m)` /
// `col(n)`, then `at(row, k)` / `at(k, col)`.
template <typename T, bool MN> struct PlainA {          // [M x K] (k contiguous) or [K x M] (m contiguous)
    static constexpr bool kFastest = !MN;
    const T* p; int64_t ld;
    using Row = const T*;
    __device__ Row row(int64_t m) const { return MN ? p + m : p + m * ld; }
    __device__ float at(Row r, int64_t k) const { return to_f32(MN ? r[k * ld] : r[k]); }
};
template <typename T, bool MN> struct PlainB {          // [N x K] (k contiguous) or [K x N] (n contiguous)
    static constexpr bool kFastest = !MN;
    const T* p; int64_t ld;
    using Col = const T*;
    __device__ Col col(int64_t n) const { return MN ? p + n : p + n * ld; }
    __device__ float at(int64_t k, Col c) const { return to_f32(MN ? c[k * ld] : c[k]); }
};
struct Pixel { int64_t b; int h, w; };
__device__ __forceinline__ Pixel pixel_of(int64_t m, int H, int W) {
    if (m >> 31) {                                           // (a 64-bit division costs some ten times a 32-bit one)
        const int64_t q = m / W;
        return Pixel{q / H, (int)(q % H), (int)(m % W)};
    }
    const unsigned u = (unsigned)m, q = u / (unsigned)W;
    return Pixel{(int64_t)(q / (unsigned)H), (int)(q % (unsigned)H), (int)(u % (unsigned)W)};
}
// k x k taps of an NHWC image as the A operand of the core's forward product: m = output pixel (b, ho, wo),
// kidx = tap * C + channel; the tap (kh, kw) of output pixel (ho, wo) is input pixel (ho * stride + kh - pad,
// wo * stride + kw - pad); pixels outside the image read as zero.
template <typename T> struct ConvFwdA {
    static constexpr bool kFastest = true;
    const T* p; ConvGeom g; int C;
    using Row = Pixel;
    __device__ Row row(int64_t m) const {
        const Pixel o = pixel_of(m, g.Ho, g.Wo);
        return Pixel{o.b, o.h * g.stride - g.pad, o.w * g.stride - g.pad};
    }
    __device__ float at(Row r, int64_t kidx) const {
        const int t = (int)kidx / C, c = (int)kidx % C, h = r.h + t / g.k, w = r.w + t % g.k;
        if (h < 0 || h >= g.H || w < 0 || w >= g.W) return 0.f;
        return to_f32(p[((r.b * g.H + h) * g.W + w) * C + c]);
    }
};
// The same taps seen from the input side, as the A operand of the data gradient: m = input pixel (b, h, w),
// kidx = tap * C + o; input pixel (h, w) met tap (kh, kw) of output pixel ((h + pad - kh) / stride,
// (w + pad - kw) / stride) where both divisions are exact and the result lies inside the output.
template <typename T> struct ConvBwdA {
    static constexpr bool kFastest = true;
    const T* p; ConvGeom g; int C;
    using Row = Pixel;
    __device__ Row row(int64_t m) const {
        const Pixel q = pixel_of(m, g.H, g.W);
        return Pixel{q.b, q.h + g.pad, q.w + g.pad};
    }
    __device__ float at(Row r, int64_t kidx) const {
        const int t = (int)kidx / C, c = (int)kidx % C;
        const int hs = r.h - t / g.k, ws = r.w - t % g.k;
        if (hs < 0 || ws < 0 || hs % g.stride || ws % g.stride) return 0.f;
        const int ho = hs / g.stride, wo = ws / g.stride;
        if (ho >= g.Ho || wo >= g.Wo) return 0.f;
        return to_f32(p[((r.b * g.Ho + ho) * g.Wo + wo) * C + c]);
    }
};
// All taps of an NHWC image as the B operand of the filter gradient: kidx = output pixel, n = tap * C + channel.
template <typename T> struct ConvTapsB {
    static constexpr bool kFastest = false;
    const T* p; ConvGeom g; int C;
    struct Col { int h, w, c; };
    __device__ Col col(int64_t n) const {
        const int t = (int)n / C;
        return Col{t / g.k - g.pad, t % g.k - g.pad, (int)n % C};
    }
    __device__ float at(int64_t kidx, Col x) const {
        const Pixel o = pixel_of(kidx, g.Ho, g.Wo);
        const int h = o.h * g.stride + x.h, w = o.w * g.stride + x.w;
        if (h < 0 || h >= g.H || w < 0 || w >= g.W) return 0.f;
        return to_f32(p[((o.b * g.H + h) * g.W + w) * C + x.c]);
    }
};
// The core G[o][tap][i] as the B operand of the data gradient: kidx = tap * Co + o, n = i.
template <typename T> struct CoreTransposedB {
    static constexpr bool kFastest = false;
    const T* p; int Ci, Co, taps;
    using Col = const T*;
    __device__ Col col(int64_t n) const { return p + n; }
    __device__ float at(int64_t kidx, Col c) const {
        const int t = (int)kidx / Co, o = (int)kidx % Co;
        return to_f32(c[((int64_t)o * taps + t) * Ci]);
    }
};

// One output tile per cluster.  A block's 256 threads form groups of GM x GN threads, each thread with RM x RN
// accumulators; the groups take every KS-th k of a tile (KS = 256 / (GM GN)) and their sums are added through shared
// memory.  The reduction is further split over the blocks of the cluster (gridDim.z), whose partial tiles are added
// through distributed shared memory: group by group and rank by rank, a fixed order.  What the small layers that land
// here wait for is latency -- a serial reduction on a handful of blocks -- so small tiles and many blocks come first,
// and the large tile, which reads shared memory least, where it fills the GPU by itself.
// 256 x 512 -> 40 in fp32: 37 us on 4 blocks of 64 x 64 without a split, 7.1 us on 16 tiles x 8 splits; forward +
// backward of the 256-token layer 139 -> 31 us.
constexpr int NT = 256, TK = 32, kMaxSplit = 8;
template <int RM_, int RN_, int GM_, int GN_> struct SimtCfg {
    static constexpr int RM = RM_, RN = RN_, GM = GM_, GN = GN_;
    static constexpr int TM = RM * GM, TN = RN * GN, KS = NT / (GM * GN);
    static constexpr int LDA = TM + 4, LDB = TN + 4;
    static constexpr int kTiles = TK * (LDA + LDB), kRed = KS * TM * TN;              // floats
    static constexpr int kSmem = (kTiles > kRed ? kTiles : kRed) + TM;                // + one column sum per row
};
using Small = SimtCfg<4, 4, 8, 8>;       // 32 x 32, four groups
using Medium = SimtCfg<4, 4, 16, 16>;    // 64 x 64
using Large = SimtCfg<8, 4, 16, 16>;     // 128 x 64

template <typename T, typename LA, typename LB> struct SimtProduct {
    int64_t M, N, K, k_per_split;
    LA la;
    LB lb;
    T* C;
    int64_t ldc;
    const T* bias;
    T* a_colsum;
};

// grid: (row tiles x column tiles of one product, then of a second one that needs nothing of the first, 1, splits)
template <typename T, typename C_, typename LA, typename LB>
__global__ void __launch_bounds__(NT, 2) simt_gemm_kernel(const __grid_constant__ SimtProduct<T, LA, LB> p0, const __grid_constant__ SimtProduct<T, LA, LB> p1, unsigned tiles0) {
    const bool second = blockIdx.x >= tiles0;
    const int64_t M = second ? p1.M : p0.M, N = second ? p1.N : p0.N, K = second ? p1.K : p0.K, k_per_split = second ? p1.k_per_split : p0.k_per_split;
    const int64_t ldc = second ? p1.ldc : p0.ldc;
    const LA la = second ? p1.la : p0.la;
    const LB lb = second ? p1.lb : p0.lb;
    T* __restrict__ C = second ? p1.C : p0.C;
    const T* __restrict__ bias = second ? p1.bias : p0.bias;
    T* __restrict__ a_colsum = second ? p1.a_colsum : p0.a_colsum;
    const unsigned tile = second ? blockIdx.x - tiles0 : blockIdx.x;
    constexpr int TM = C_::TM, TN = C_::TN, KS = C_::KS, RM = C_::RM, RN = C_::RN, LDA = C_::LDA, LDB = C_::LDB;
    constexpr int FA = TM * TK / NT, FB = TN * TK / NT;      // elements of each operand a thread brings in per tile
    __shared__ __align__(16) float smem[C_::kSmem];
    float* As = smem;
    float* Bs = smem + TK * LDA;
    ptx::griddep_wait();
    ptx::griddep_launch_dependents();       // (in this order: see GemmArgs::a_early)
    const int t = threadIdx.x;
    const int64_t n_tiles = (N + TN - 1) / TN;
    const int64_t m0 = (int64_t)(tile / n_tiles) * TM, n0 = (int64_t)(tile % n_tiles) * TN;
    const int64_t k_begin = (int64_t)blockIdx.z * k_per_split, k_end = k_begin + k_per_split < K ? k_begin + k_per_split : K;
    const int grp = t / (C_::GM * C_::GN), gt = t % (C_::GM * C_::GN);
    const int tx = gt % C_::GN, ty = gt / C_::GN;            // thread computes rows ty * RM .., columns tx * RN .. of its group
    constexpr bool ak = LA::kFastest, bk = LB::kFastest;
    const bool sums = a_colsum && n0 == 0;                   // this tile column also adds up A over k
    float acc[RM][RN] = {};
    float csum = 0.f;                                        // of row t % TM, the k of this thread's share
    // Where a thread's elements of a tile lie: 16 k x 16 rows per pass where k is the contiguous index, else TM (TN)
    // rows x NT / TM k per pass.
    constexpr int AR = ak ? TM / 16 : 1, BR = bk ? TN / 16 : 1;
    typename LA::Row arow[AR];
    typename LB::Col bcol[BR];
    const int64_t m_last = M - 1, n_last = N - 1;
#pragma unroll
    for (int i = 0; i < AR; ++i) { const int64_t m = m0 + (ak ? t / 16 + 16 * i : t % TM); arow[i] = la.row(m < M ? m : m_last); }
#pragma unroll
    for (int i = 0; i < BR; ++i) { const int64_t n = n0 + (bk ? t / 16 + 16 * i : t % TN); bcol[i] = lb.col(n < N ? n : n_last); }
    // The next tile's elements are fetched into registers before the current tile is multiplied: their global-memory
    // latency then runs beside the arithmetic instead of in front of it (the order of the additions is unchanged).
    float ra[FA], rb[FB];
    auto fetch = [&](int64_t k0) {
#pragma unroll
        for (int i = 0; i < FA; ++i) {
            const int mm = ak ? t / 16 + 16 * (i % AR) : t % TM, kk = ak ? t % 16 + 16 * (i / AR) : t / TM + NT / TM * i;
            ra[i] = (m0 + mm < M && k0 + kk < k_end) ? la.at(arow[i % AR], k0 + kk) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < FB; ++i) {
            const int nn = bk ? t / 16 + 16 * (i % BR) : t % TN, kk = bk ? t % 16 + 16 * (i / BR) : t / TN + NT / TN * i;
            rb[i] = (n0 + nn < N && k0 + kk < k_end) ? lb.at(k0 + kk, bcol[i % BR]) : 0.f;
        }
    };
    if (k_begin < k_end) fetch(k_begin);
    for (int64_t k0 = k_begin; k0 < k_end; k0 += TK) {
#pragma unroll
        for (int i = 0; i < FA; ++i) {
            const int mm = ak ? t / 16 + 16 * (i % AR) : t % TM, kk = ak ? t % 16 + 16 * (i / AR) : t / TM + NT / TM * i;
            As[kk * LDA + mm] = ra[i];
        }
#pragma unroll
        for (int i = 0; i < FB; ++i) {
            const int nn = bk ? t / 16 + 16 * (i % BR) : t % TN, kk = bk ? t % 16 + 16 * (i / BR) : t / TN + NT / TN * i;
            Bs[kk * LDB + nn] = rb[i];
        }
        __syncthreads();
        if (k0 + TK < k_end) fetch(k0 + TK);
        if (sums) {
            constexpr int per = TK / (NT / TM);
            const int m = t % TM, kk0 = t / TM * per;
#pragma unroll
            for (int i = 0; i < per; ++i) csum += As[(kk0 + i) * LDA + m];
        }
#pragma unroll
        for (int kq = 0; kq < TK / KS; ++kq) {
            const int kk = kq * KS + grp;
            float a[RM], b[RN];
#pragma unroll
            for (int i = 0; i < RM; i += 4) {
                const float4 x = *reinterpret_cast<const float4*>(&As[kk * LDA + ty * RM + i]);
                a[i] = x.x; a[i + 1] = x.y; a[i + 2] = x.z; a[i + 3] = x.w;
            }
#pragma unroll
            for (int j = 0; j < RN; j += 4) {
                const float4 x = *reinterpret_cast<const float4*>(&Bs[kk * LDB + tx * RN + j]);
                b[j] = x.x; b[j + 1] = x.y; b[j + 2] = x.z; b[j + 3] = x.w;
            }
#pragma unroll
            for (int i = 0; i < RM; ++i)
#pragma unroll
                for (int j = 0; j < RN; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
    auto put = [&](int64_t m, int64_t n, float v) {
        if (bias) v += to_f32(bias[n]);
        C[m * ldc + n] = from_f32<T>(v);
    };
    const int S = (int)gridDim.z;
    if (KS == 1 && S == 1) {                                 // nothing to add up: straight from the registers
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
            for (int j = 0; j < RN; ++j) {
                const int64_t m = m0 + ty * RM + i, n = n0 + tx * RN + j;
                if (m < M && n < N) put(m, n, acc[i][j]);
            }
    }
    float* csums = smem + C_::kSmem - TM;
    if (sums) {                                              // the shares of a row, added in ascending order
        smem[t] = csum;                                      // (the tiles are dead)
        __syncthreads();
        if (t < TM) {
            float x = 0.f;
#pragma unroll
            for (int i = 0; i < NT / TM; ++i) x += smem[i * TM + t];
            csums[t] = x;
        }
        __syncthreads();
    }
    if (KS > 1 || S > 1) {
        // The groups' sums are added in this block first and the blocks' sums are fetched all at once: read one after the other out of
        // the peers' shared memory, 32 of them behind one another cost more than the products.  fp32 passes: 512 -> 512 at rank 40,
        // 256 tokens 23.6 -> 21.9 us; 520 -> 264 at 96, 76 tokens 23.2 -> 17.0; 536 -> 600 at 178, 510 tokens 64.2 -> 60.1.
        float* red = smem;                                   // [KS][TM][TN], then [TM][TN]
#pragma unroll
        for (int i = 0; i < RM; ++i)
#pragma unroll
            for (int j = 0; j < RN; j += 4)
                *reinterpret_cast<float4*>(&red[(grp * TM + ty * RM + i) * TN + tx * RN + j]) = make_float4(acc[i][j], acc[i][j + 1], acc[i][j + 2], acc[i][j + 3]);
        if (KS > 1) {
            __syncthreads();
            for (int e = 4 * t; e < TM * TN; e += 4 * NT) {
                float4 v = *reinterpret_cast<const float4*>(&red[e]);
#pragma unroll
                for (int q = 1; q < KS; ++q) {
                    const float4 x = *reinterpret_cast<const float4*>(&red[q * TM * TN + e]);
                    v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
                }
                *reinterpret_cast<float4*>(&red[e]) = v;     // (read and written by this thread alone)
            }
        }
        cg::cluster_group cluster = cg::this_cluster();
        if (S > 1) cluster.sync(); else __syncthreads();
        const int rank = S > 1 ? (int)cluster.block_rank() : 0;
        for (int e = rank * NT + t; e < TM * TN; e += S * NT) {
            const int64_t m = m0 + e / TN, n = n0 + e % TN;
            if (m >= M || n >= N) continue;
            float x[kMaxSplit];
#pragma unroll
            for (int z = 0; z < kMaxSplit; ++z) x[z] = z < S ? (S > 1 ? cluster.map_shared_rank(red, z) : red)[e] : 0.f;
            float v = x[0];
#pragma unroll
            for (int z = 1; z < kMaxSplit; ++z) v += x[z];
            put(m, n, v);
        }
        if (sums && rank == 0 && t < TM && m0 + t < M) {
            float x[kMaxSplit], v = 0.f;
#pragma unroll
            for (int z = 0; z < kMaxSplit; ++z) x[z] = z < S ? (S > 1 ? cluster.map_shared_rank(csums, z) : csums)[t] : 0.f;
#pragma unroll
            for (int z = 0; z < kMaxSplit; ++z) v += x[z];
            a_colsum[m0 + t] = from_f32<T>(v);
        }
        if (S > 1) cluster.sync();                           // no block leaves while a peer still reads its partial tile
    } else if (sums && t < TM && m0 + t < M) {
        a_colsum[m0 + t] = from_f32<T>(csums[t]);
    }
}

// Two-stage column sum for tall matrices: stage 1 adds the rows of one of S row ranges for 64 columns
// (4 row lanes per column, fixed order), stage 2 adds the S partial rows in ascending order.
template <typename T>
__global__ void __launch_bounds__(256) colsum_stage1_kernel(const T* __restrict__ A, int64_t lda, int64_t M, int64_t N,
                                                            int64_t rows_per_split, float* __restrict__ partial) {
    __shared__ float part[4][64];
    const int c = threadIdx.x % 64, g = threadIdx.x / 64;
    const int64_t n = (int64_t)blockIdx.x * 64 + c;
    const int64_t m_begin = (int64_t)blockIdx.y * rows_per_split;
    const int64_t m_end = m_begin + rows_per_split < M ? m_begin + rows_per_split : M;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    if (n < N) {
        int64_t m = m_begin + g;
        for (; m + 12 < m_end; m += 16) {          // four independent loads in flight per thread
            s0 += to_f32(A[m * lda + n]);
            s1 += to_f32(A[(m + 4) * lda + n]);
            s2 += to_f32(A[(m + 8) * lda + n]);
            s3 += to_f32(A[(m + 12) * lda + n]);
        }
        for (; m < m_end; m += 4) s0 += to_f32(A[m * lda + n]);
    }
    part[g][c] = (s0 + s1) + (s2 + s3);
    __syncthreads();
    if (g == 0 && n < N) partial[(int64_t)blockIdx.y * N + n] = (part[0][c] + part[1][c]) + (part[2][c] + part[3][c]);
}

template <typename T>
__global__ void __launch_bounds__(256) colsum_stage2_kernel(const float* __restrict__ partial, int splits, int64_t N,
                                                            T* __restrict__ out) {
    const int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    float tot = 0.f;
    for (int z = 0; z < splits; ++z) tot += partial[(int64_t)z * N + n];
    out[n] = from_f32<T>(tot);
}

template <typename T>
lrd_status_t colsum_two_stage_t(const void* A, int64_t lda, int64_t M, int64_t N, void* out, float* scratch, int splits,
                                cudaStream_t stream) {
    const int64_t rows = (M + splits - 1) / splits;
    dim3 grid((unsigned)((N + 63) / 64), (unsigned)splits);
    colsum_stage1_kernel<T><<<grid, 256, 0, stream>>>((const T*)A, lda, M, N, rows, scratch);
    colsum_stage2_kernel<T><<<(unsigned)((N + 255) / 256), 256, 0, stream>>>(scratch, splits, N, (T*)out);
    count_launch(2);
    return cudaGetLastError() == cudaSuccess ? LRD_OK : LRD_ERR_CUDA;
}

// Tile and split.  A block's time is its fused multiply-adds (per thread and k: RM RN of them, and the shared-memory reads
// around them: the small tile runs at about half the rate of the large one) plus some 3000 clocks of loads, sums and
// stores; two blocks share an SM.  The reduction is split while the grid has fewer than two blocks per SM and a share
// still has 32 k.
struct SimtPlan { int cfg, splits; double clocks; };
constexpr int kTileM[3] = {128, 64, 32}, kTileN[3] = {64, 64, 32};
int64_t simt_tiles(int cfg, int64_t M, int64_t N) { return ((M + kTileM[cfg] - 1) / kTileM[cfg]) * ((N + kTileN[cfg] - 1) / kTileN[cfg]); }
SimtPlan simt_plan(int64_t M, int64_t N, int64_t K, int64_t M1 = 0, int64_t N1 = 0, int64_t K1 = 0) {
    const double per_k[3] = {90.0, 48.0, 18.0};              // clocks of a block per k
    SimtPlan best{2, 1, 1e300};
    const int64_t deep = K > K1 ? K : K1, shallow = M1 > 0 && K1 < K ? K1 : K;
    for (int c = 0; c < 3; ++c) {
        const int64_t tiles = simt_tiles(c, M, N) + (M1 > 0 ? simt_tiles(c, M1, N1) : 0);
        for (int S = 1; S <= kMaxSplit; ++S) {
            if (S > 1 && (tiles * S > 2 * kNumSms || (shallow + S - 1) / S < TK)) break;
            const double waves = (double)((tiles * S + 2 * kNumSms - 1) / (2 * kNumSms));
            const double share = (double)((deep + S - 1) / S);
            const double crowd = tiles * S > kNumSms ? 1.6 : 1.0;                       // two blocks on an SM share its units
            const double cost = waves * (share * per_k[c] * crowd + 3000.0 + (S > 1 ? 1200.0 : 0.0));
            if (cost < best.clocks) best = {c, S, cost};
        }
    }
    return best;
}

// One product, or two independent ones (p1) in one launch.
template <typename T, typename Cfg, typename LA, typename LB>
lrd_status_t simt_launch(int splits, SimtProduct<T, LA, LB> p0, const SimtProduct<T, LA, LB>* second, cudaStream_t stream) {
    SimtProduct<T, LA, LB> p1 = second ? *second : p0;
    auto tiles = [](const SimtProduct<T, LA, LB>& p) { return (unsigned)(((p.N + Cfg::TN - 1) / Cfg::TN) * ((p.M + Cfg::TM - 1) / Cfg::TM)); };
    for (auto* p : {&p0, &p1}) p->k_per_split = ((p->K + splits - 1) / splits + TK - 1) / TK * TK;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(tiles(p0) + (second ? tiles(p1) : 0u), 1, (unsigned)splits);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the kernel waits (griddepcontrol.wait) before it touches global memory
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = (unsigned)splits;
    cfg.attrs = attr;
    cfg.numAttrs = splits > 1 ? 2 : 1;
    if (!cuda_ok(cudaLaunchKernelEx(&cfg, simt_gemm_kernel<T, Cfg, LA, LB>, p0, p1, tiles(p0)), "cudaLaunchKernelEx(general product)"))
        return LRD_ERR_CUDA;
    count_launch();
    return LRD_OK;
}

template <typename T, typename LA, typename LB>
lrd_status_t simt_run(const SimtPlan& pl, const SimtProduct<T, LA, LB>& p0, const SimtProduct<T, LA, LB>* p1, cudaStream_t s) {
    switch (pl.cfg) {
        case 0:  return simt_launch<T, Large>(pl.splits, p0, p1, s);
        case 1:  return simt_launch<T, Medium>(pl.splits, p0, p1, s);
        default: return simt_launch<T, Small>(pl.splits, p0, p1, s);
    }
}

template <typename T, typename LA, typename LB>
lrd_status_t simt_product(int64_t M, int64_t N, int64_t K, const LA& la, const LB& lb, void* C, int64_t ldc, const void* bias, void* a_colsum,
                          cudaStream_t s) {
    const SimtProduct<T, LA, LB> p{M, N, K, 0, la, lb, (T*)C, ldc, (const T*)bias, (T*)a_colsum};
    return simt_run<T, LA, LB>(simt_plan(M, N, K), p, nullptr, s);
}

template <typename T>
lrd_status_t simt_wgrad_pair_t(const SimtPlan& pl, const GemmArgs& a, const GemmArgs& b, cudaStream_t s) {
    using P = SimtProduct<T, PlainA<T, true>, PlainB<T, true>>;
    auto product = [](const GemmArgs& g) {
        return P{g.M, g.N, g.K, 0, PlainA<T, true>{(const T*)g.A, g.lda}, PlainB<T, true>{(const T*)g.B, g.ldb}, (T*)g.C, g.ldc, (const T*)g.bias, (T*)g.a_colsum};
    };
    const P p0 = product(a), p1 = product(b);
    return simt_run<T, PlainA<T, true>, PlainB<T, true>>(pl, p0, &p1, s);
}

template <typename T>
lrd_status_t simt_gemm_t(const GemmArgs& g, cudaStream_t stream) {
    const T *A = (const T*)g.A, *B = (const T*)g.B;
    auto run = [&](const auto& la, const auto& lb) { return simt_product<T>(g.M, g.N, g.K, la, lb, g.C, g.ldc, g.bias, g.a_colsum, stream); };
    if (g.a_mn_major)
        return g.b_mn_major ? run(PlainA<T, true>{A, g.lda}, PlainB<T, true>{B, g.ldb}) : run(PlainA<T, true>{A, g.lda}, PlainB<T, false>{B, g.ldb});
    return g.b_mn_major ? run(PlainA<T, false>{A, g.lda}, PlainB<T, true>{B, g.ldb}) : run(PlainA<T, false>{A, g.lda}, PlainB<T, false>{B, g.ldb});
}

template <typename T>
lrd_status_t conv_fwd_t(const void* in, const void* G, void* out, int64_t B, const ConvGeom& g, int ci, int co, cudaStream_t stream) {
    // M = output pixels, N = co, K = taps * ci, B = G as [co x taps * ci] (k contiguous)
    const int64_t P = B * g.Ho * g.Wo, K = (int64_t)g.k * g.k * ci;
    return simt_product<T>(P, co, K, ConvFwdA<T>{(const T*)in, g, ci}, PlainB<T, false>{(const T*)G, K}, out, co, nullptr, nullptr, stream);
}

template <typename T>
lrd_status_t conv_bwd_data_t(const void* dout, const void* G, void* din, int64_t B, const ConvGeom& g, int ci, int co,
                             cudaStream_t stream) {
    // M = input pixels, N = ci, K = taps * co, B = G regrouped as (tap, o) x i
    const int64_t P = B * g.H * g.W, K = (int64_t)g.k * g.k * co;
    return simt_product<T>(P, ci, K, ConvBwdA<T>{(const T*)dout, g, co}, CoreTransposedB<T>{(const T*)G, ci, co, g.k * g.k}, din, ci, nullptr, nullptr, stream);
}

template <typename T>
lrd_status_t conv_filter_t(const void* dout, const void* in, void* dG, int64_t B, const ConvGeom& g, int ci, int co,
                           cudaStream_t stream) {
    // M = co, N = taps * ci, K = output pixels
    const int64_t P = B * g.Ho * g.Wo, N = (int64_t)g.k * g.k * ci;
    return simt_product<T>(co, N, P, PlainA<T, true>{(const T*)dout, co}, ConvTapsB<T>{(const T*)in, g, ci}, dG, N, nullptr, nullptr, stream);
}

}  // namespace

lrd_status_t simt_gemm(const GemmArgs& g, cudaStream_t stream) {
    if (g.M <= 0 || g.N <= 0) return LRD_OK;
    return g.dtype == LRD_F32 ? simt_gemm_t<float>(g, stream) : simt_gemm_t<__nv_bfloat16>(g, stream);
}

// Two weight gradients that need nothing of each other: one launch where that is estimated to be faster, as it is while neither
// fills the GPU (512 -> 512 at rank 40, 256 tokens, fp32, forward and backward: 31.4 us in six launches, 25.4 in five).
lrd_status_t simt_wgrads(const GemmArgs& a, const GemmArgs& b, cudaStream_t s) {
    const bool alike = a.dtype == b.dtype && a.a_mn_major && a.b_mn_major && b.a_mn_major && b.b_mn_major && a.M > 0 && a.N > 0 && b.M > 0 && b.N > 0;
    if (alike) {
        const SimtPlan pl = simt_plan(a.M, a.N, a.K, b.M, b.N, b.K);
        if (pl.clocks < simt_plan(a.M, a.N, a.K).clocks + simt_plan(b.M, b.N, b.K).clocks)
            return a.dtype == LRD_F32 ? simt_wgrad_pair_t<float>(pl, a, b, s) : simt_wgrad_pair_t<__nv_bfloat16>(pl, a, b, s);
    }
    const lrd_status_t st = simt_gemm(a, s);
    return st != LRD_OK ? st : simt_gemm(b, s);
}

lrd_status_t simt_conv_fwd(const void* in, const void* G, void* out, int64_t B, const ConvGeom& g, int64_t ci, int64_t co,
                           lrd_dtype_t dt, cudaStream_t s) {
    return dt == LRD_F32 ? conv_fwd_t<float>(in, G, out, B, g, (int)ci, (int)co, s)
                         : conv_fwd_t<__nv_bfloat16>(in, G, out, B, g, (int)ci, (int)co, s);
}
lrd_status_t simt_conv_bwd_data(const void* dout, const void* G, void* din, int64_t B, const ConvGeom& g, int64_t ci,
                                int64_t co, lrd_dtype_t dt, cudaStream_t s) {
    return dt == LRD_F32 ? conv_bwd_data_t<float>(dout, G, din, B, g, (int)ci, (int)co, s)
                         : conv_bwd_data_t<__nv_bfloat16>(dout, G, din, B, g, (int)ci, (int)co, s);
}
lrd_status_t simt_conv_bwd_filter(const void* dout, const void* in, void* dG, int64_t B, const ConvGeom& g, int64_t ci,
                                  int64_t co, lrd_dtype_t dt, cudaStream_t s) {
    return dt == LRD_F32 ? conv_filter_t<float>(dout, in, dG, B, g, (int)ci, (int)co, s)
                         : conv_filter_t<__nv_bfloat16>(dout, in, dG, B, g, (int)ci, (int)co, s);
}

int colsum_splits(int64_t M) {
    int64_t s = M / 64;
    return (int)(s < 1 ? 1 : (s > 64 ? 64 : s));
}

}  // namespace lrd

// ---- bias gradient without any caller-provided or allocated scratch -----------------------------------
// The partial column sums of the two-stage kernels live in a file-scope device array, so a caller
// that may not allocate device memory can still get the many-block version.
namespace {

constexpr int64_t kNoAllocMaxN = 8192;                           // widest dY this entry point accepts
constexpr int kNoAllocMaxSplits = 64;
constexpr size_t kNoAllocFloats = (size_t)kNoAllocMaxN * kNoAllocMaxSplits;   // 2 MiB per GPU that loads the library
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocFloats];

constexpr int kNoallocMaxDevices = 64;
float* g_noalloc_ptr[kNoallocMaxDevices] = {};                          // device address of the array, per device

// In host code `g_noalloc_scratch` is only a handle for the runtime, not an address a kernel can use:
// the device address is asked for once per device (with that device current) and cached.
lrd_status_t noalloc_scratch(float** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoallocMaxDevices) return LRD_ERR_CUDA;
    if (!g_noalloc_ptr[dev]) {
        float* ptr = nullptr;
        if (cudaGetSymbolAddress((void**)&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return LRD_ERR_CUDA;
        g_noalloc_ptr[dev] = ptr;
    }
    *out = g_noalloc_ptr[dev];
    return LRD_OK;
}

}  // namespace

extern "C" lrd_status_t lrd_bias_grad_noalloc(const void* dY, int64_t ldy, int64_t M, int64_t N, void* dbias,
                                              lrd_dtype_t dtype, void* cuda_stream) {
    if (M < 0 || N < 1 || (dtype != LRD_F32 && dtype != LRD_BF16)) return LRD_ERR_INVALID_ARG;
    if (!dbias || (M > 0 && !dY)) return LRD_ERR_INVALID_ARG;
    if (ldy == 0) ldy = N;
    if (ldy < N) return LRD_ERR_INVALID_ARG;
    if (N > kNoAllocMaxN) return LRD_ERR_TOO_LARGE;
    const size_t e = lrd::elem_size(dtype);
    if (((uintptr_t)dbias % e) || ((uintptr_t)dY % e)) return LRD_ERR_ALIGNMENT;
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess)
        return LRD_ERR_CUDA;
    if (major != 10) return LRD_ERR_ARCH;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    if (M == 0) return cudaMemsetAsync(dbias, 0, (size_t)N * e, stream) == cudaSuccess ? LRD_OK : LRD_ERR_CUDA;
    float* scratch = nullptr;
    const lrd_status_t st = noalloc_scratch(&scratch);
    if (st != LRD_OK) return st;
    // At most 64 splits, so the partial sums fit; stage 1 writes every partial that stage 2 reads, so nothing left by an earlier call is ever used.
    const int splits = lrd::colsum_splits(M);
    return dtype == LRD_F32 ? lrd::colsum_two_stage_t<float>(dY, ldy, M, N, dbias, scratch, splits, stream)
                            : lrd::colsum_two_stage_t<__nv_bfloat16>(dY, ldy, M, N, dbias, scratch, splits, stream);
}
