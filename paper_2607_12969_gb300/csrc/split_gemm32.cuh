// split_gemm32.cuh -- products of binary32 matrices on the tensor cores
// (split_gemm32.cu): operands and the product itself.
#pragma once

#include "common.cuh"

namespace lrc {
namespace sg32 {

constexpr int kParts = 3;          // bfloat16 parts of a binary32 value
constexpr int kKB = 16;            // columns of the reduction per image block
constexpr int kGroupBytes = kParts * 8 * kKB * 2;      // 8 rows of one block
constexpr int kNTMax = 256;
// Rows of the second side a tile takes: split reductions share the rows evenly
// (a multiple of 16); else 256, or 128 where that pads less (the epilogue's
// stores take 32 columns of a quarter of the tile at a time).
inline int n_tile(int64_t rows, bool splitk) {
    if (!splitk) return (rows + 127) / 128 % 2 ? 128 : 256;
    const int64_t tiles = (rows + kNTMax - 1) / kNTMax;
    return (int)(((rows + tiles - 1) / tiles + 15) / 16 * 16);
}

// One operand of a product, `rows` x K: entry (r, c) is p[r rs + c cs]; `second`
// the side it is on.  The image is [block of kKB columns][group of 8 rows][part][column octet][8 rows x
// 16 bytes] and serves as either side of a product.
struct Operand {
    const float* p;
    int64_t rs, cs, rows, K;
    bool second;
    unsigned char* img;
    int* hard;               // hard[0] = rows the parts cannot carry, hard[1 ...] their indices, then a mark per row
};
inline int64_t image_rows(int64_t rows) { return (rows + 255) / 256 * 256; }
inline int64_t image_blocks(int64_t K) { return (K + kKB - 1) / kKB; }
inline size_t image_bytes(int64_t rows, int64_t K) { return (size_t)(image_rows(rows) / 8) * image_blocks(K) * kGroupBytes; }
inline size_t hard_bytes(int64_t rows) { return ((size_t)(2 * rows + 1) * 4 + 255) & ~(size_t)255; }

// Parts of up to three operands, in one launch.  The row lists have been set
// to zero (all of their bytes).
lrc_status split(const Operand* const* ops, int count, cudaStream_t s);

// C(i, j) at C[i ldc + j]: the product A B^T times cscale[j] (may be null; null
// with `splitk` false).  `splitk` splits the reduction over the CTAs (few, deep
// tiles); its partial sums, part_bytes() of them at `part`, are added in a fixed
// order.  Rows that the parts cannot carry are recomputed with binary32 FMAs.
size_t part_bytes(int64_t M, int64_t N);
lrc_status product(const Operand& A, const Operand& B, float* C, int64_t ldc, const float* cscale, bool splitk,
                   float* part, cudaStream_t s);

}  // namespace sg32
}  // namespace lrc
