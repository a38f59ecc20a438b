// Host-side construction of TMA tensor maps.  The driver's encoder is reached through the
// runtime's entry-point query, so the library links against the CUDA runtime only.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace lrd {

// 2-D bf16 tensor [rows x cols], row stride ld elements, box [box_rows x box_cols]; the swizzle
// span equals the box row (128, 64 or 32 bytes; none otherwise, or where asked for); zero fill outside the tensor.
// Returns false on failure.
bool make_tmap_2d_bf16(CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols, uint64_t ld_elems,
                       uint32_t box_rows, uint32_t box_cols, bool swizzled = true);

// 4-D bf16 NHWC tensor [B][H][W][C], box [1][box_h][box_w][box_c], 128-byte swizzle, zero fill.
bool make_tmap_nhwc_bf16(CUtensorMap* out, const void* base, uint64_t B, uint64_t H, uint64_t W, uint64_t C,
                         uint32_t box_h, uint32_t box_w, uint32_t box_c);

// bf16 NHWC tensor [B][H][W][C] in im2col mode: a load fetches `pixels` consecutive positions of a sliding window (w
// fastest, then h, then the image), 64 channels of each, 128-byte swizzle, zero fill outside the image.  The window's
// first tap visits columns low_w, low_w + step, ... (n_w of them) and rows low_h, low_h + step, ... (n_h).
bool make_tmap_im2col_bf16(CUtensorMap* out, const void* base, uint64_t B, uint64_t H, uint64_t W, uint64_t C, int low_h, int low_w,
                           int n_h, int n_w, int step, uint32_t pixels);

}  // namespace lrd
