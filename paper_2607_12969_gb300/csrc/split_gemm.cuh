// split_gemm.cuh -- products of binary64 matrices on the tensor cores
// (split_gemm.cu): operands, images and the product itself.
#pragma once

#include "common.cuh"

namespace lrc {
namespace sg {

constexpr int kParts64 = 7;        // 9-bit digits a binary64 value is cut into
constexpr int kKB = 16;            // columns of the reduction per image block
constexpr int64_t kMaxK = 1 << 20; // longest reduction the 64-bit sums hold
constexpr int kStatSplits = 128;    // most slices of the reduction in the row statistics

// Tiles of the product: 128 rows of the first side, and of the second the rows
// split evenly over tiles of at most kNTMax, a multiple of 16.
constexpr int kNTMax = 64;
inline int n_tile(int64_t rows) {
    const int64_t tiles = (rows + kNTMax - 1) / kNTMax;
    return (int)(((rows + tiles - 1) / tiles + 15) / 16 * 16);
}

// A matrix whose rows are cut into digits: entry (r, c) is p[r rs + c cs]
// times 2^(sh sign) with sh half the exponent of scale[c] (scale may be null).
// For W = (X V) diag(s) and U of a second product W U^T with scale = s and
// signs -1 and +1: with s_j decaying over many orders the entries of a row of
// W would lie far below its first ones; this halves that distance on either
// side, exactly.
struct Src64 {
    const double* p;
    int64_t rs, cs;
    const double* scale;
    int sign;
};

// One operand of a product, `rows` x K, and its digits.  The image is
// [block of kKB columns][group of 8 rows][digit][column octet][8 rows x 16
// bytes]: the blocks of any run of row groups are contiguous, so the same image
// serves as either side of a product, with tiles of any height.
struct Operand64 {
    Src64 src;
    int64_t rows, K;
    unsigned char* img;      // digits
    int* exps;               // exponent of every row (image rows)
    unsigned char* kind;     // what every row's digits are (split_gemm.cu)
    int* stats;              // row statistics per slice of K
};
constexpr int kMaxOps = 5;   // operands per slice()

constexpr int kGroupBytes = kParts64 * 8 * kKB * 2;      // one row group of one block
// Rows are padded to 16; a tile that reaches past them reads the next block's
// first rows (or the kTailBytes behind the image), which only reach entries
// that are not stored.
inline int64_t image_rows(int64_t rows) { return (rows + 15) / 16 * 16; }
constexpr int kTailBytes = 16 * kGroupBytes;
inline int64_t image_blocks(int64_t K) { return (K + kKB - 1) / kKB; }
size_t operand_bytes(int64_t rows, int64_t K);
// Carves an operand's buffers out of `ws` (256-byte aligned).
void operand_carve(Operand64* o, unsigned char* ws);

// Digits of up to kMaxOps operands (at most two launches for all of them).
// clear[0 ... nclear), at most 256 counters, are set to zero on the way.
lrc_status slice(const Operand64* const* ops, int count, int* clear, int nclear, cudaStream_t s);

// Blocks of a product that may hold entries which the digits do not carry: `list`
// holds fix_bytes(M, N) for an M x N product, *count is zero before it.
struct Fix {
    int2* list;
    int* count;
};
size_t fix_bytes(int64_t M, int64_t N);

// C(i, j) at C[i cr + j cc], i < A.rows, j < B.rows: the product A B^T times
// rscale[i] cscale[j] (each may be null, and both are with `split` false).  `split` splits the reduction over
// the CTAs (few, deep tiles); its partial sums are added in a fixed order.
// `part` holds part_bytes() bytes.  Entries that the digits do not carry are
// recomputed with binary64 FMAs.
struct Out64 {
    double* C;
    int64_t cr, cc;
    const double* rscale;
    const double* cscale;
};
size_t part_bytes(int64_t M, int64_t N);
// Columns of the tiles that an M x N product takes.
int product_tile(int64_t M, int64_t N);
lrc_status product(const Operand64& A, const Operand64& B, const Out64& out, bool split, double* part, const Fix& fix,
                   cudaStream_t s);
// C(i, j) = C(j, i) at C[i ldc + j]: A A^T, `part` and `fix` as above.  Tiles
// below the diagonal are left out.
lrc_status gram(const Operand64& A, double* C, int64_t ldc, double* part, const Fix& fix, cudaStream_t s);

}  // namespace sg
}  // namespace lrc
