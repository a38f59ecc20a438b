// Shared host/device declarations of the library (internal).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lrd.h"

namespace lrd {

// Per-device host-side caches (function attributes set, occupancy answers, symbol addresses) are kept in tables
// indexed by the current device's ordinal; devices past the table share its last row.
constexpr int kMaxDevices = 16;
inline int device_slot() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
    return dev < kMaxDevices ? dev : kMaxDevices - 1;
}

// Device address (on the current device) of the flag a bounded wait raises when it runs out (one word, zero = fine);
// nullptr if the address cannot be obtained.  Read and cleared by lrd_check_device_status().
unsigned int* device_timeout_flag();
lrd_status_t read_and_clear_device_timeout(bool* raised);
// One block whose bounded wait is left to run out (see lrd_selftest_wait_timeout).
lrd_status_t selftest_wait_runs_out(cudaStream_t stream);

// One matrix product  C[M x N] = op(A) op(B) (+ bias over columns), fp32 accumulate.
//   a_mn_major = false: A stored [M x K] (k contiguous);  true: A stored [K x M] (m contiguous)
//   b_mn_major = false: B stored [N x K] (k contiguous);  true: B stored [K x N] (n contiguous)
struct GemmArgs {
    int64_t M, N, K;
    const void* A; int64_t lda; bool a_mn_major;
    const void* B; int64_t ldb; bool b_mn_major;
    void* C; int64_t ldc;
    const void* bias;          // [N] or nullptr, same dtype as C
    void* a_colsum = nullptr;  // optional [M]: sum over k of A(m, k) (the bias gradient when A is dY); both operands MN-major
    lrd_dtype_t dtype;         // storage type of A, B, C, bias
    int max_cluster_split = 0; // split weight gradients: largest cluster to split the reduction over (0 = automatic).  A
                               // launch meant to run BESIDE others asks for 2: clusters of 4 or 8 need that many free
                               // SMs inside one GPC, which a chain kernel on 128 of the 148 SMs never leaves
    bool add = false;          // weight gradients on the tensor-core kernels: C (and a_colsum) += the product, rounded to the storage
                               // type before the fp32 sum and after it
    bool whole = false;        // data products: the reduction is not split over a cluster
    // Weight gradients on the single-SM kernels, and B of data products on the persistent one: this operand is loaded without waiting
    // for the launch before this one (griddepcontrol.wait).  Two things have to hold.  Between the start of the call and this
    // launch stands one that lets the next launch start only behind its own wait: all data passes (both chains, the data products,
    // convolutions, the one-launch pass, the general products) do, weight gradients (both kernels) and copies that are early
    // themselves let it start before, and are nothing to rely on.  What the call found in memory is complete by then.  And neither that launch nor a later
    // one of the call writes the operand.  Every launch waits for the one before it before it ends, early ones too, so that whoever
    // waits for the last has waited for all.  A launch boundary costs some 1.5 us behind the last block's exit and another for the
    // first loads.
    // Gradients: 768 -> 768 at r = 192, a pass over 128 tokens 18.5 -> 17.7 us, over 4096 26.3 -> 25.7; six layers of 768 (4096
    // tokens) replayed 170.8 -> 168.6.
    bool a_early = false, b_early = false;
    bool any_rows = false;     // weight gradients: C of any stride and alignment (single-SM kernels)
    bool in_turn = false;      // weight gradients: started only when the launch before has ended (blocks that wait on an SM for
                               // that end keep it from work in other streams)
};

// True when the CUDA call succeeded.  With the environment variable LRD_LOG_ERRORS set, a failure is also written to
// stderr with the call's name and CUDA's error string (the C ABI itself only returns LRD_ERR_CUDA).
bool cuda_ok(cudaError_t e, const char* what);

// Host-side count of kernels enqueued (see lrd_launch_count).
void count_launch(int n = 1);

inline size_t elem_size(int dtype) { return dtype == LRD_BF16 ? 2 : 4; }
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// General fp32-FMA path (any shape, any alignment).
lrd_status_t simt_gemm(const GemmArgs& g, cudaStream_t stream);
lrd_status_t simt_wgrads(const GemmArgs& a, const GemmArgs& b, cudaStream_t s);

// One product on the path chosen by `path` (an lrd_path_t): the tensor-core kernel when the
// operands qualify, else the general kernel.
lrd_status_t run_gemm(const GemmArgs& g, int path, bool allow_split, float* partials, size_t partial_bytes,
                      cudaStream_t s);
// Several weight gradients (reduction split as above), independent of one another; their scratch may be shared.
lrd_status_t run_wgrads(const GemmArgs* g, int n, int path, float* const* partials, const size_t* partial_bytes, cudaStream_t s);
GemmArgs make_gemm(int64_t M, int64_t N, int64_t K, const void* A, int64_t lda, bool a_mn, const void* B, int64_t ldb,
                   bool b_mn, void* C, int64_t ldc, const void* bias, lrd_dtype_t dt);
lrd_status_t zero_fill(void* p, int64_t rows, int64_t cols, int64_t ld, lrd_dtype_t dt, cudaStream_t s);
// One matrix of a repacking launch: dst[0 .. rows_dst)[0 .. cols_dst) = src where it has that row and column, else zero;
// bf16, any leading dimensions and alignments.
struct Copy2d {
    void* dst; int64_t ldd;
    const void* src; int64_t lds;
    int64_t rows_src, rows_dst;
    int cols_src, cols_dst;
};
constexpr int kMaxCopies = 6;
// All of them in one launch.  Sources must not overlap destinations.  early: nothing of them is written by, or read by, the launch
// before this one (see GemmArgs::a_early).
lrd_status_t copy2d_bf16(const Copy2d* c, int n, cudaStream_t s, bool early = false);

}  // namespace lrd
