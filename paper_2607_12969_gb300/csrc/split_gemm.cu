// split_gemm.cu -- binary64 products C = A B^T on the tensor cores.
//
// This GPU multiplies bfloat16 numbers on its tensor cores about 1300 times
// as fast as it multiplies binary64 numbers (1.26 TFLOP/s), so a binary64
// product is formed from exact products of short pieces (the error-free
// splitting of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and
// its applications", Numer. Algorithms 59, 2012):
//
//   * every row of A and of B is scaled by a power of two to at most 1/2 and
//     cut into seven signed 9-bit digits d_0 ... d_6 (|d_0| <= 128, |d_i| <=
//     256), x = 2^(e - 7) sum_i d_i 2^(-9 i): 62 bits below the row's largest
//     entry, so entries down to 2^-9 of it are carried without error.  A
//     digit is a bfloat16 number.
//   * C = sum over classes t = i + j of 2^(-9 t) D_i E_j^T, each class in an
//     accumulator of its own.  Within 64 terms of the reduction the sums of
//     classes 0 to 4 are integers of at most 2^20, 2^22, 2^23, 2^23.6 and
//     2^24, so the tensor cores' binary32 accumulation forms them without
//     error; those of classes 5 and 6 are as a rule, and where not the error
//     is 2^-24 of a class that lies 2^-45 below the first.  Classes from 7 on
//     are left out (28 products of 49).
//   * every 64 terms (`period`: less often where the bound allows) the
//     accumulators are drained into two 64-bit integers per entry, and the
//     whole sum is rounded to binary64 once.
//
// The error, in units of B_i B_j (B: the power of two above a row's largest
// entry), is as a rule below 2^-61 a term with a sign of its own, and at worst
// about 2^-57 a term, where the digits are all at their limits and of one sign
// (the six products of class 7 alone then reach 2^-58.4).  That is small beside
// S_ij = sum_k |a_ik b_jk| unless the large entries of one row meet zeros or
// small entries of the other, where binary64 FMAs would be more exact.  So
// S_ij is estimated from the first digits, sum_k |d_0 e_0| 2^-14, and an entry
// of C for which that stays below 2^-5 (kMinSum) is listed and recomputed by
// binary64 FMAs (repair_kernel).  The others are as a rule within
// 0.1 sqrt(K) 2^-53 S_ij, and at worst (first digits rounded up from halves
// besides) within K 2^-50 S_ij; FMA sums of K terms are bounded by K 2^-53 S_ij.
// Rows of Gaussian entries reach the limit within 16 terms for all but 1e-6 of
// the entries, also with columns scaled by j^-1.5 or 0.9^j.  Where one of the rows
// has first digits only (units, signs, small integers) no class is left out, the
// other row's rounding (2^-62 of its B a term) is all there is, and the limit is
// 2^-9 (kMinShort).
//
// Rows that hold an infinity, a NaN or a largest entry outside 2^-480 ...
// 2^495 get zero digits, so that all their entries are listed.
//
// Kernels: row statistics (row_stats_kernel), digits (slice_kernel, which
// writes them as images that either side of a product loads by bulk copies),
// the product and the estimates of S (product_kernel, persistent, one CTA a
// SM), the ordered sum of split reductions (part_sum_kernel) and the
// recomputed entries (repair_kernel).
#include <algorithm>
#include <utility>

#include "split_gemm.cuh"
#include "split_pieces.cuh"
#include "tc.cuh"

namespace lrc {
namespace sg {

namespace {

using namespace tc;

__device__ unsigned int g_err_split;

constexpr int64_t kOwnStatsK = 512;    // reductions up to this long: slice_kernel takes the row statistics itself
constexpr int kNonFinite = 1 << 20;    // marks a row with an infinity or NaN in its statistics
constexpr int kNoEntry = -(1 << 20);   // ... one without nonzero entries
// Kinds of rows: with digits past the first; with first digits only; with none,
// because it holds nothing but zeros, or because the digits cannot carry it.
enum RowKind : unsigned char { kDeepRow, kShortRow, kZeroRow, kHardRow };
constexpr float kMinSum = 512.0f, kMinShort = 32.0f;     // 2^-5 and 2^-9 in units of products of first digits
// Biased exponents of a row's largest entry that digits carry: with both rows
// inside, every result is zero or a normal number (round_pq).
constexpr int kMinExp = 544, kMaxExp = 1518;

// ---------------------------------------------------------------- sources
struct View64 {
    Src64 s;
    __device__ double at(int64_t r, int64_t k) const { return __ldg(s.p + r * s.rs + k * s.cs); }
    __device__ int shift(int64_t k) const {
        if (!s.scale) return 0;
        const int e = (int)((uint64_t)__double_as_longlong(__ldg(s.scale + k)) >> 52) & 0x7ff;
        return e == 0 || e == 0x7ff ? 0 : s.sign * ((e - 1023) / 2);
    }
};

// Biased exponent of |x| (bits), a subnormal's as if the range went on; x != 0.
__device__ __forceinline__ int biased_exp(uint64_t bits) {
    const int e = (int)(bits >> 52) & 0x7ff;
    if (e != 0) return e == 0x7ff ? kNonFinite : e;
    return 12 - __clzll((long long)(bits & 0xfffffffffffffull));
}

// ---------------------------------------------------------------- statistics
// The largest biased exponent of a row's nonzero entries.
__device__ __forceinline__ void stat_add(int& mx, double x, int shift) {
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu, e = h >> 20;
    int v = (int)e + shift;
    if (e - 1u >= 0x7feu) {            // zero, subnormal, infinity or NaN
        const uint32_t lo = (uint32_t)__double2loint(x);
        v = (h | lo) != 0 ? biased_exp(((uint64_t)h << 32) | lo) + shift : kNoEntry;
    }
    mx = max(mx, v);
}

// What the kernels below take of an operand, and its share of the blocks.
struct Job {
    View64 v;
    int64_t rows, K, img_rows, kblocks;
    int64_t b0;              // first block
    int64_t kchunk;          // columns a block takes
    int kparts, splits, vec;
    int* stats;              // splits > 0: statistics per slice of K; else slice_kernel takes its own
    unsigned char* img;
    int* exps;
    unsigned char* kind;
};
struct Jobs {
    Job j[kMaxOps];
    int n;
    int nclear;
    int* clear;              // counters to set to zero
};
__device__ __forceinline__ const Job& job_of(const Jobs& js, int64_t block) {
    int i = 0;
    while (i + 1 < js.n && block >= js.j[i + 1].b0) ++i;
    return js.j[i];
}

// Statistics of 32 rows over columns [k0, k1), by 256 threads; row r0 + lane's
// in warp 0.  K contiguous: a warp per row, lanes along K; else a lane per
// row, so that either way a warp reads consecutive addresses.
template <bool SCALED>
__device__ __forceinline__ int block_stats(const View64& v, int64_t r0, int64_t rows, int64_t k0, int64_t k1, bool vec,
                                           int (&sm)[8][32]) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto shift = [&](int64_t k) { return SCALED ? v.shift(k) : 0; };
    if (v.s.cs == 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t r = r0 + warp + 8 * q;
            int a = kNoEntry;
            if (r < rows) {
                int64_t k = k0 + 2 * lane;
                if (vec) {
                    for (; k + 194 <= k1; k += 256) {
                        double2 x[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            x[u] = __ldg(reinterpret_cast<const double2*>(v.s.p + r * v.s.rs + k + 64 * u));
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            stat_add(a, x[u].x, shift(k + 64 * u));
                            stat_add(a, x[u].y, shift(k + 64 * u + 1));
                        }
                    }
                }
                for (; k < k1; k += 64) {
                    stat_add(a, v.at(r, k), shift(k));
                    if (k + 1 < k1) stat_add(a, v.at(r, k + 1), shift(k + 1));
                }
            }
            a = __reduce_max_sync(0xffffffffu, a);
            if (lane == 0) sm[0][warp + 8 * q] = a;
        }
    } else {
        const int64_t r = r0 + lane;
        int a = kNoEntry;
        if (r < rows) {
            int64_t k = k0 + warp;
            for (; k + 24 < k1; k += 32) {
                double x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = v.at(r, k + 8 * u);
#pragma unroll
                for (int u = 0; u < 4; ++u) stat_add(a, x[u], shift(k + 8 * u));
            }
            for (; k < k1; k += 8) stat_add(a, v.at(r, k), shift(k));
        }
        sm[warp][lane] = a;
    }
    __syncthreads();
    int t = kNoEntry;
    if (warp == 0) {
        t = sm[0][lane];
        if (v.s.cs != 1) {
#pragma unroll
            for (int w = 1; w < 8; ++w) t = max(t, sm[w][lane]);
        }
    }
    return t;
}

__global__ void __launch_bounds__(256, 6) row_stats_kernel(const __grid_constant__ Jobs js) {
    __shared__ int sm[8][32];
    pdl_wait();
    pdl_trigger();
    const Job& o = job_of(js, blockIdx.x);
    const int64_t lb = (int64_t)blockIdx.x - o.b0, rg = lb / o.splits, z = lb - rg * o.splits;
    const int64_t r0 = rg * 32, k0 = z * o.kchunk;
    if (blockIdx.x == 0 && threadIdx.x < js.nclear) js.clear[threadIdx.x] = 0;
    const int64_t k1 = min(o.K, k0 + o.kchunk);
    const int a = o.v.s.scale ? block_stats<true>(o.v, r0, o.rows, k0, k1, o.vec != 0, sm)
                              : block_stats<false>(o.v, r0, o.rows, k0, k1, o.vec != 0, sm);
    if (threadIdx.x < 32 && r0 + threadIdx.x < o.rows) {
        o.stats[z * o.rows + r0 + threadIdx.x] = a;
        if (z == 0) o.kind[r0 + threadIdx.x] = kShortRow;
    }
}

// ---------------------------------------------------------------- digits
// The seven digits of eight values as bfloat16: w[p][q] holds digits
// p of values 2q (low half) and 2q + 1.  em: biased exponent of the row's
// largest entry.  The value is rounded to a multiple of 2^-61 of 2^(em -
// 1022), the power of two above it, and the digits are those of that integer
// plus 256 at every place but the first, minus 256 again: a number read with
// digits in [-256, 255].  `any` collects the integers' bits.
__device__ __forceinline__ void digits8(const double (&x)[8], const int (&sh)[8], int em, uint32_t (&w)[kParts64][4],
                                        uint64_t& any) {
    constexpr uint64_t kBias =
        256ull * (1ull + (1ull << 9) + (1ull << 18) + (1ull << 27) + (1ull << 36) + (1ull << 45));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float f[2][kParts64];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t b = __double_as_longlong(x[2 * q + h]);
            const int e = (int)((uint64_t)b >> 52) & 0x7ff;
            const int64_t mant = (b & 0xfffffffffffffll) | (e ? (1ll << 52) : 0);
            const int s = (e ? e : 1) + sh[2 * q + h] - em + 8;      // <= 8
            int64_t v;
            if (s >= 0) v = mant << s;
            else v = s > -55 ? (mant + (1ll << (-s - 1))) >> -s : 0;
            if (b < 0) v = -v;
            any |= (uint64_t)v;
            const uint64_t t = (uint64_t)v + kBias;
            const int d0 = (int)((int64_t)t >> 54);
            f[h][0] = __int_as_float(0x4b400000 + d0) - 12582912.0f;
#pragma unroll
            for (int i = 1; i < kParts64; ++i) {
                const uint32_t d = (uint32_t)(t >> (9 * (6 - i))) & 511u;
                f[h][i] = __int_as_float(0x4b400000u | d) - (12582912.0f + 256.0f);
            }
        }
#pragma unroll
        for (int i = 0; i < kParts64; ++i)
            w[i][q] = __byte_perm(__float_as_uint(f[0][i]), __float_as_uint(f[1][i]), 0x7632);
    }
}

// Digits into the image (split_gemm.cuh).  A CTA takes 32 image rows
// and `kchunk` columns (of an operand with a short reduction all of them, and
// takes the row statistics itself); a lane is a row, so that a warp's 16-byte
// stores of one digit are four runs of 128 bytes.
__global__ void __launch_bounds__(256, 4) slice_kernel(const __grid_constant__ Jobs js) {
    __shared__ int sm[8][32];
    __shared__ int s_em[32], s_deep[32];
    pdl_wait();
    pdl_trigger();
    const Job& o = job_of(js, blockIdx.x);
    const View64 v = o.v;
    const int64_t rows = o.rows, K = o.K;
    const int64_t lb = (int64_t)blockIdx.x - o.b0, rg = lb / o.kparts, kp = lb - rg * o.kparts;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t r0 = rg * 32;
    int own = kNoEntry;
    if (o.splits == 0) own = block_stats<true>(v, r0, rows, 0, K, o.vec != 0, sm);
    if (tid < 32) {
        const int64_t r = r0 + lane;
        int mx = own;
        if (r < rows)
            for (int z = 0; z < o.splits; ++z) mx = max(mx, o.stats[(int64_t)z * rows + r]);
        const bool none = r >= rows || mx == kNoEntry, hard = !none && (mx < kMinExp || mx > kMaxExp);
        s_em[lane] = none || hard ? -1 : mx;
        s_deep[lane] = 0;
        if (kp == 0 && r < o.img_rows) {
            o.exps[r] = none || hard ? 1023 : mx;
            if (none || hard) o.kind[r] = none ? kZeroRow : kHardRow;
        }
    }
    __syncthreads();
    const int64_t r = r0 + lane;
    const int em = s_em[lane];
    uint64_t any = 0;
    const size_t block_bytes = (size_t)(o.img_rows / 8) * kGroupBytes;
    unsigned char* row_base = o.img + (size_t)(r >> 3) * kGroupBytes + (r & 7) * 16;
    const int64_t o1 = r < o.img_rows ? min((kp + 1) * o.kchunk, o.kblocks * kKB) / 8 : 0;
    for (int64_t oc = kp * o.kchunk / 8 + warp; oc < o1; oc += 8) {
        double x[8];
        int sh[8];
        const int64_t k0 = oc * 8;
        if (em < 0) {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = 0.0;
        } else if (o.vec && k0 + 8 <= K) {
            const double2* p = reinterpret_cast<const double2*>(v.s.p + r * v.s.rs + k0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const double2 d = __ldg(p + j);
                x[2 * j] = d.x;
                x[2 * j + 1] = d.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = k0 + j < K ? v.at(r, k0 + j) : 0.0;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) sh[j] = (v.s.scale && k0 + j < K) ? v.shift(k0 + j) : 0;
        uint32_t w[kParts64][4];
        digits8(x, sh, em < 0 ? 1023 : em, w, any);
        unsigned char* dst = row_base + (size_t)(oc >> 1) * block_bytes + (size_t)(oc & 1) * 128;
#pragma unroll
        for (int i = 0; i < kParts64; ++i)
            *reinterpret_cast<uint4*>(dst + i * (8 * kKB * 2)) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
    }
    if (any & ((1ull << 54) - 1)) s_deep[lane] = 1;        // digits past the first
    __syncthreads();
    if (tid < 32 && r < rows && em >= 0) {
        // (row_stats_kernel has made it kShortRow where several CTAs have a part of the row)
        if (s_deep[lane]) o.kind[r] = kDeepRow;
        else if (o.splits == 0) o.kind[r] = kShortRow;
    }
}

// ---------------------------------------------------------------- product
constexpr int kMaxListed = 120;
struct GemmArgs {
    const unsigned char* A;
    const unsigned char* B;
    const int* ea;
    const int* eb;
    double* C;               // split: partial tiles [slot][column][128 rows]
    int64_t cr, cc, M, N;
    int ntiles, tiles;       // tiles of B; all tiles
    int chunks;              // 64-column chunks of the reduction
    int kblocks;             // 16-column blocks
    int split, group, stages, tma;
    int64_t a_block, b_block;    // bytes of a block of either image
    uint32_t a_bytes, b_bytes;   // of a tile's part of it
    int2* fix;                   // listed blocks (first row, first column), and their number
    int* nfix;
    int listed;                  // > 0: the tiles are list[0 ... listed), row << 8 | column
    uint16_t list[kMaxListed];
    uint32_t tmem_cols;
};

// Sixteen epilogue warps, four per quarter of the tensor-memory lanes, each
// with a quarter of the columns: with eight, two a scheduler, the drain's and
// the rounding's dependent steps were not covered (a 128 x 64 tile of two
// chunks took 26000 clocks, its MMAs 10750).
constexpr int kEpiWarps = 16;
constexpr int kThreads = 32 * (4 + kEpiWarps);
// Registers: the first four warps (producer, MMA issuer, two that estimate the
// sums of magnitudes) hand some
// of theirs to the epilogue's, which keep two 64-bit sums per entry: 128 x 64
// + 512 x 104 = 61440, the 640 x 96 = 61440 of the launch.
constexpr int kRegsLow = 64, kRegsEpi = 104;
// Row and column of a tile.
__device__ __forceinline__ int2 tile_at(const GemmArgs& a, int tile) {
    if (a.listed) return make_int2(a.list[tile] >> 8, a.list[tile] & 255);
    const int mt = tile / a.ntiles;
    return make_int2(mt, tile - mt * a.ntiles);
}

constexpr int kChunkBlocks = 64 / kKB;
constexpr uint32_t kCtrlBytes = 1024;
constexpr int kStageBytes = 32 * 64;           // a warp's rows on their way out

// Chunks between drains of a class's accumulator: its sums stay at most 2^24
// (classes 5 and 6: see above).  A converting drain costs an entry 8 clocks of
// a scheduler's F2I rate per class and chunk.
__host__ __device__ constexpr int period(int t) { return t == 0 ? 16 : t == 2 ? 2 : t == 3 || t == 4 ? 1 : 4; }

__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[8]) { tmem_ld8(taddr, r); }
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t (&r)[4]) { tmem_ld4(taddr, r); }

// Adds HC columns of an accumulator, times `weight`, to the sums.
template <int HC>
__device__ __forceinline__ void drain(uint32_t taddr, int weight, int64_t (&sum)[HC]) {
    constexpr int G = HC % 8 == 0 ? 8 : 4;
    uint32_t v[HC / G][G];
#pragma unroll
    for (int q = 0; q < HC / G; ++q) tmem_ld_cols(taddr + q * G, v[q]);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < HC; ++j) sum[j] += (int64_t)__float2int_rn(__uint_as_float(v[j / G][j % G])) * weight;
}

// Classes 5 and 6 together, in units of 2^-4 of class 5's.
template <int HC>
__device__ __forceinline__ void drain56(uint32_t t5, uint32_t t6, int64_t (&sum)[HC]) {
    constexpr int G = 4;
#pragma unroll
    for (int q = 0; q < HC; q += G) {
        uint32_t u[G], v[G];
        tmem_ld_cols(t5 + q, u);
        tmem_ld_cols(t6 + q, v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < G; ++j)
            sum[q + j] += __float2int_rn(fmaf(__uint_as_float(v[j]), 0.03125f, __uint_as_float(u[j]) * 16.0f));
    }
}

// P 2^-27 + Q 2^-49 times 2^(esum - 2058), rounded to nearest; esum is the sum
// of the biased exponents of the two rows' largest entries (a row's value is
// its digit sum times 2^(e - 1029)).  |P| < 2^63, |Q| < 2^62; the sum's
// integer, in units of 2^-59, is below 2^95 (reductions of up to 2^20 terms),
// so kMinExp and kMaxExp keep the result's exponent within 1 ... 2046.
// Straight-line code, so that a thread's entries interleave: it runs on the
// integer pipe, at half an instruction a clock, and with K = 128 takes about
// as long per tile as the MMAs.
__device__ __forceinline__ double round_pq(int64_t p, int64_t q, int esum) {
    p += q >> 22;
    uint32_t a = (uint32_t)((uint64_t)p >> 32), b = (uint32_t)p, c = (uint32_t)q << 10;
    const uint32_t neg = (uint32_t)((int32_t)a >> 31);
    a ^= neg;
    b ^= neg;
    c ^= neg;
    asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;" : "+r"(c), "+r"(b), "+r"(a) : "r"(neg));
    int n = esum - 1000;
#pragma unroll
    for (int z = 0; z < 2; ++z) {
        const bool up = a == 0;
        a = up ? b : a;
        b = up ? c : b;
        c = up ? 0 : c;
        n -= up ? 32 : 0;
    }
    const int s = __clz((int)a);
    const uint32_t e = a ? (uint32_t)(n - s) << 20 : 0u;       // (exponent - 1) << 20; a == 0: the sum is zero
    const uint32_t hi = __funnelshift_l(b, a, s), mid = __funnelshift_l(c, b, s);
    uint32_t r0 = __funnelshift_r(mid, hi, 11), r1 = hi >> 11, t = mid << 21;
    // + the first bit dropped (to nearest, ties away from zero)
    asm("add.cc.u32 %2, %2, %2;\n\taddc.cc.u32 %0, %0, 0;\n\taddc.u32 %1, %1, %3;" : "+r"(r0), "+r"(r1), "+r"(t) : "r"(e));
    return __hiloint2double((int)(r1 | (neg & 0x80000000u)), (int)r0);
}

// The same through two binary64 additions: p' = p + (q >> 22) and the rest of q
// as binary64 numbers by their encodings, 1.5 2^52 + p' and 2^30 + rest 2^-22,
// added with the constants' sum taken off first (exact).  For |p'| < 2^51.  The
// binary64 pipe takes 128 clocks of a scheduler for it, the integer pipe about
// 80 for round_pq, so the epilogue gives three entries of eight to it.
__device__ __forceinline__ double round_pq_fp64(int64_t p, int64_t q, int esum) {
    p += q >> 22;
    const double a = __hiloint2double((int)((uint64_t)p >> 32) + 0x43380000, (int)p);
    const double b = __hiloint2double(0x41d00000, (int)((uint32_t)q & 0x3fffffu));
    const double y = __dadd_rn(__dsub_rn(a, 6755399441055744.0 + 1073741824.0), b);
    const int hi = __double2hiint(y);
    return __hiloint2double(hi ? hi + ((esum - 2085) << 20) : 0, __double2loint(y));
}

// The products of classes [T0, T1) of one block from digit I of A on,
// straight-line (a branch between two MMAs costs about as much as one).  All
// that share a digit of A follow one another: A stays in the collector buffer
// (an MMA of 64 columns is bound by its reads of shared memory, 48 clocks with
// A's 4 KB read and 35 with them kept), and no MMA adds to the accumulator of
// the one before it, which would wait for its result (about 120 clocks).
// fresh: bit t is set where class t starts a new sum.
// col3: column of class 3's accumulator.
template <int NT, int T0, int T1, int I = 0, int J = (T0 > 0 ? T0 : 0)>
__device__ __forceinline__ void issue(uint32_t tmem, uint32_t col3, uint32_t fresh, uint32_t alo, uint32_t ahi,
                                      uint32_t blo, uint32_t bhi) {
    constexpr int kPart = 8 * kKB * 2 / 16;                                     // one digit
    constexpr int J0 = T0 > I ? T0 - I : 0, J1 = T1 - I;                        // digits of B for this one of A
    constexpr int kMmaUse = J1 - J0 == 1 ? kNoReuse : J == J0 ? kFill : J == J1 - 1 ? kLast : kUse;
    mma_f16_col<kMmaUse>(tmem + (I + J == 3 ? col3 : (uint32_t)(I + J) * NT), alo + I * kPart, ahi, blo + J * kPart, bhi,
                          idesc_f16_f32(128, NT) | kIdescBF16, I > 0 ? 1u : ((fresh >> (I + J)) & 1u) ^ 1u);
    if constexpr (J + 1 < J1) issue<NT, T0, T1, I, J + 1>(tmem, col3, fresh, alo, ahi, blo, bhi);
    else if constexpr (I + 1 < T1) issue<NT, T0, T1, I + 1, (T0 > I + 1 ? T0 - I - 1 : 0)>(tmem, col3, fresh, alo, ahi,
                                                                                                  blo, bhi);
}

// Four bytes of an image's first digits: those of row `lane` / 4 of a group and
// columns 2 (lane % 4) + {0, 1} of an octet, without their signs.
__device__ __forceinline__ uint32_t first_digits(const unsigned char* group, int octet, int lane) {
    return __ldg(reinterpret_cast<const uint32_t*>(group + octet * 128 + lane * 4)) & 0x7fff7fffu;
}
// The same as an A fragment of m16n8k16: two row groups, both octets.
__device__ __forceinline__ void first_digits_a(const unsigned char* p, int lane, uint32_t (&d)[4]) {
    d[0] = first_digits(p, 0, lane);
    d[1] = first_digits(p + kGroupBytes, 0, lane);
    d[2] = first_digits(p, 1, lane);
    d[3] = first_digits(p + kGroupBytes, 1, lane);
}
// d = a b + c (16 x 8, 16 terms)
__device__ __forceinline__ void mma_16x8(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2],
                                         float c0, float c1, float c2, float c3) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
                 "{%8, %9}, {%10, %11, %12, %13};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(c0), "f"(c1), "f"(c2), "f"(c3));
}

// Lists the blocks (16 rows, half a tile's columns) in which an entry's sum of
// magnitudes, estimated from the first digits of the first 16 terms, does not reach
// kMinSum; repair_kernel looks at those more closely.  Straight from the images,
// whose octets have the layout of m16n8k16 fragments.  Two warps have the time of a
// tile's MMAs and epilogue for this, if the loads are not waited for one by one and
// the registers that the first warps keep suffice (16384 x 8192, k = 128, b = 8192:
// 1577 us without the estimates, 2016 with each load waited for, 1616 with the
// longer sums here too).
template <int NT>
__device__ __forceinline__ void list_small_sums(const GemmArgs& a, int mt, int nt, int half, int lane) {
    constexpr int J = NT / 16, kBatch = 4;
    constexpr uint32_t kBeyond = 0x49804980u;              // 2^20, twice: past the edges every sum is large
    const int row_t = mt * 128, col0 = nt * NT + half * (NT / 2);
    if (col0 >= a.N) return;
    uint32_t b[J][2];
    {
        const unsigned char* p = a.B + (int64_t)(col0 >> 3) * kGroupBytes;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const bool in = col0 + 8 * j + (lane >> 2) < a.N;
            b[j][0] = in ? first_digits(p + j * kGroupBytes, 0, lane) : kBeyond;
            b[j][1] = in ? first_digits(p + j * kGroupBytes, 1, lane) : kBeyond;
        }
    }
    uint32_t failed = 0;
    for (int s0 = 0; s0 < 8; s0 += kBatch) {
        const unsigned char* rows = a.A + (int64_t)((row_t >> 3) + 2 * s0) * kGroupBytes;
        uint32_t x[kBatch][4];
#pragma unroll
        for (int s = 0; s < kBatch; ++s)                   // (rows are padded to 16)
            if (row_t + 16 * (s0 + s) < a.M) first_digits_a(rows + s * 2 * kGroupBytes, lane, x[s]);
#pragma unroll
        for (int s = 0; s < kBatch; ++s) {
            const int row0 = row_t + 16 * (s0 + s);
            if (row0 >= a.M) break;
            if (row0 + 16 > a.M) {
                if (row0 + (lane >> 2) >= a.M) x[s][0] = x[s][2] = kBeyond;
                if (row0 + (lane >> 2) + 8 >= a.M) x[s][1] = x[s][3] = kBeyond;
            }
            float acc[J][4], least;
#pragma unroll
            for (int j = 0; j < J; ++j) mma_16x8(acc[j], x[s], b[j], 0.0f, 0.0f, 0.0f, 0.0f);
            least = acc[0][0];
#pragma unroll
            for (int j = 0; j < J; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) least = fminf(least, acc[j][i]);
            failed |= __all_sync(0xffffffffu, least >= kMinSum) ? 0u : 1u << (s0 + s);
        }
    }
    if (lane == 0 && failed) {
        int2* list = a.fix + atomicAdd(a.nfix, __popc(failed));
        for (; failed; failed &= failed - 1) *list++ = make_int2(row_t + 16 * (__ffs((int)failed) - 1), col0);
    }
}

template <int NT>
__global__ void __launch_bounds__(kThreads, 1) product_kernel(const __grid_constant__ GemmArgs a,
                                                              const __grid_constant__ CUtensorMap tm_c) {
    constexpr int HC = NT / 4;          // columns a thread drains
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + 8;
    uint64_t* gfull = empty + 8;        // classes 0 to 3 of an even or odd chunk complete; classes 4 to 6
    uint64_t* gempty = gfull + 3;       // ... drained
    uint64_t* mma_done = gempty + 3;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    unsigned char* ring = smem + kCtrlBytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t stage_bytes = a.a_bytes + a.b_bytes;
    unsigned int* err = &g_err_split;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 3; ++i) {
            mbar_init(&gfull[i], 1);
            mbar_init(&gempty[i], 32 * kEpiWarps);
        }
        mbar_init(mma_done, 1);
        *abort = 0;
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc(tmem_slot, a.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    pdl_wait();
    pdl_trigger();

    if (warp >= 4) {
        reg_inc<kRegsEpi>();
        // ------------------------------------------------------------ epilogue
        const int g = warp & 3, quarter = (warp - 4) >> 2;      // of the lanes, of the columns
        const uint32_t tbase = tmem + ((uint32_t)(g * 32) << 16) + quarter * HC;
        const int r = g * 32 + lane;
        unsigned char* stage = ring + (size_t)a.stages * stage_bytes + (size_t)(warp - 4) * kStageBytes;
        Pieces<GemmArgs> pc(a);
        int tile, c0, c1;
        int ch = 0;
        bool ok = true;
        // One lane of a warp polls (512 polling threads would take the MMA issuer's
        // issue slots), and the warps do not wait for one another: while one drains,
        // on the conversion and FMA pipes, another rounds, on the integer pipe.
        auto epi_wait = [&](uint64_t* bar, uint32_t parity) {
            bool got = true;
            if (lane == 0) got = mbar_wait(bar, parity, abort, err, 4u);
            return __all_sync(0xffffffffu, got) != 0;
        };
        while (ok && pc.next(a, &tile, &c0, &c1)) {
            const int2 at = tile_at(a, tile);
            const int mt = at.x, nt = at.y;
            const int64_t row = (int64_t)mt * 128 + r, col0 = (int64_t)nt * NT + quarter * HC;
            // exponents: of the thread's row, and of column `lane`
            const int ea = row < a.M ? a.ea[row] : 0;
            const int eb = lane < HC && col0 + lane < a.N ? a.eb[col0 + lane] : 0;
            int64_t P[HC], Q[HC];
#pragma unroll
            for (int j = 0; j < HC; ++j) P[j] = Q[j] = 0;
            for (int c = c0; c < c1; ++c, ++ch) {
                const int n = c - c0 + 1;
                auto due = [&](int t) { return c + 1 == c1 || n % period(t) == 0; };
                if (!(ok = epi_wait(&gfull[ch & 1], (ch >> 1) & 1))) break;
                tc_fence_after();
                drain<HC>(tbase + (ch & 1 ? 7 : 3) * NT, 1, P);
                if (due(2)) drain<HC>(tbase + 2 * NT, 1 << 9, P);
                if (due(1)) drain<HC>(tbase + NT, 1 << 18, P);
                if (due(0)) drain<HC>(tbase, 1 << 27, P);
                tc_fence_before();
                mbar_arrive(&gempty[ch & 1]);
                if (!(ok = epi_wait(&gfull[2], ch & 1))) break;
                tc_fence_after();
                drain<HC>(tbase + 4 * NT, 1 << 13, Q);
                if (due(5)) drain56<HC>(tbase + 5 * NT, tbase + 6 * NT, Q);
                tc_fence_before();
                mbar_arrive(&gempty[2]);
            }
            if (!ok) break;
            if (a.split) {
                double* dst = a.C + part_slot(a, tile) * (128 * NT) + (int64_t)(quarter * HC) * 128 + r;
#pragma unroll
                for (int j = 0; j < HC; ++j) dst[j * 128] = round_pq(P[j], Q[j], ea + __shfl_sync(0xffffffffu, eb, j));
                continue;
            }
            const bool shallow = a.chunks <= 8;      // |P| stays below 2^50
            auto value = [&](int j) {
                const int es = ea + __shfl_sync(0xffffffffu, eb, j);
                return shallow && ((0x52 >> (j & 7)) & 1) ? round_pq_fp64(P[j], Q[j], es) : round_pq(P[j], Q[j], es);
            };
            if (a.cc == 1) {
                // 32 rows x CG columns at a time through shared memory (64-byte rows in
                // the 64-byte swizzle, or 32-byte rows) and out by TMA, or where a row's pitch does
                // not allow that by runs of CG: stores straight from the registers, 32
                // bytes a row, filled the load/store unit
                constexpr int CG = HC % 8 == 0 ? 8 : 4;
#pragma unroll
                for (int j0 = 0; j0 < HC; j0 += CG) {
                    double y[CG];
#pragma unroll
                    for (int j = 0; j < CG; ++j) y[j] = value(j0 + j);
                    if (a.tma && lane == 0) bulk_wait_read<0>();      // the store before has read the buffer
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < CG; j += 2) {
                        const int c = CG == 8 ? (j >> 1) ^ ((lane >> 1) & 3) : j >> 1;
                        *reinterpret_cast<double2*>(stage + lane * (CG * 8) + c * 16) = make_double2(y[j], y[j + 1]);
                    }
                    const int64_t rb = (int64_t)mt * 128 + g * 32;
                    if (a.tma) {
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0 && rb < a.M && col0 + j0 < a.N) {
                            tma_store_2d(&tm_c, (int32_t)(col0 + j0), (int32_t)rb, stage);
                            bulk_commit();
                        }
                    } else {
                        __syncwarp();
                        const int q = lane % CG, r0 = lane / CG;
                        double* dst = a.C + (rb + r0) * a.cr + col0 + j0 + q;
                        const bool mine = col0 + j0 + q < a.N;
#pragma unroll
                        for (int i = 0; i < CG; ++i) {
                            const int rr = i * (32 / CG) + r0;
                            const int c = CG == 8 ? (q >> 1) ^ ((rr >> 1) & 3) : q >> 1;
                            const double d = *reinterpret_cast<const double*>(stage + rr * (CG * 8) + c * 16 + (q & 1) * 8);
                            if (mine && rb + rr < a.M) dst[(int64_t)i * (32 / CG) * a.cr] = d;
                        }
                    }
                }
            } else {
                double* dst = a.C + row * a.cr + col0 * a.cc;
#pragma unroll
                for (int j = 0; j < HC; ++j) {
                    const double y = value(j);
                    if (row < a.M && col0 + j < a.N) dst[j * a.cc] = y;
                }
            }
        }
        if (a.tma && lane == 0) bulk_wait<0>();
    } else {
        reg_dec<kRegsLow>();
        if (warp == 0) {
            // ------------------------------------------------------------ producer
            if (lane == 0) {
                Pieces<GemmArgs> pc(a);
                int tile, c0, c1;
                int it = 0, slot = 0;
                uint32_t phase = 1;
                bool ok = true;
                while (ok && pc.next(a, &tile, &c0, &c1)) {
                    const int2 at = tile_at(a, tile);
                    const int mt = at.x, nt = at.y;
                    const int b1 = min(kChunkBlocks * c1, a.kblocks);
                    for (int kb = kChunkBlocks * c0; kb < b1; ++kb, ++it) {
                        if (!(ok = mbar_wait(&empty[slot], phase, abort, err, 1u))) break;
                        unsigned char* dst = ring + (size_t)slot * stage_bytes;
                        mbar_arrive_expect_tx(&full[slot], stage_bytes);
                        bulk_load(dst, a.A + kb * a.a_block + (size_t)mt * a.a_bytes, a.a_bytes, &full[slot]);
                        bulk_load(dst + a.a_bytes, a.B + kb * a.b_block + (size_t)nt * a.b_bytes, a.b_bytes, &full[slot]);
                        if (++slot == a.stages) {
                            slot = 0;
                            phase ^= 1;
                        }
                    }
                }
                if (!ok) {
                    volatile int no_abort = 0;
                    for (int j = it - a.stages > 0 ? it - a.stages : 0; j < it; ++j)
                        mbar_wait(&full[j % a.stages], (j / a.stages) & 1, &no_abort, err, 0u, 100000000ull);
                }
            }
        } else if (warp == 1) {
            // ------------------------------------------------------------ MMA issuer
            // The whole warp walks the loop and waits; one lane issues, in one branch
            // per block (with a branch or an election per MMA the warp, which shares
            // its scheduler with busy epilogue warps, issued one in 49 to 100 clocks).
            Pieces<GemmArgs> pc(a);
            int tile, c0, c1;
            int slot = 0, ch = 0;
            uint32_t phase = 0;            // parity of the ring's current pass
            bool ok = true;
            // waits agree on every lane before the warp goes on
            auto wait = [&](uint64_t* bar, uint32_t parity) {
                return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort, err, 2u)) != 0;
            };
            // column octets 128 bytes apart, row groups kGroupBytes
            const uint64_t ad = smem_desc(smem_u32(ring), 128, kGroupBytes, 0);
            const uint64_t bd = smem_desc(smem_u32(ring) + a.a_bytes, 128, kGroupBytes, 0);
            const uint32_t ahi = (uint32_t)(ad >> 32), bhi = (uint32_t)(bd >> 32), alo0 = (uint32_t)ad, blo0 = (uint32_t)bd;
            while (ok && pc.next(a, &tile, &c0, &c1)) {
                for (int c = c0; c < c1 && ok; ++c, ++ch) {
                    const int nb = min(kChunkBlocks, a.kblocks - kChunkBlocks * c);
                    uint32_t fresh = 0;
#pragma unroll
                    for (int t = 0; t < kParts64; ++t) fresh |= (c - c0) % period(t) == 0 ? 1u << t : 0u;
                    // Classes 0 to 3 of the whole chunk, drained while the others run.  Class
                    // 3, the only one of them drained every chunk, has two accumulators, so
                    // the chunk waits for the drain before the last one, and for the last
                    // one only where it emptied one of classes 0 to 2 (128 x 64 tiles of two
                    // chunks: the second chunk's MMAs no longer wait for the rounding and
                    // stores of the tile before).
                    if (!(ok = wait(&gempty[ch & 1], ((ch >> 1) & 1) ^ 1))) break;
                    if ((fresh & 7) && ch > 0 && !(ok = wait(&gempty[(ch - 1) & 1], ((ch - 1) >> 1) & 1))) break;
                    const uint32_t col3 = (uint32_t)(ch & 1 ? 7 : 3) * NT;
                    for (int b0 = 0; b0 < nb; b0 += 2) {
                        // two blocks per wait, half the lanes polling each
                        const int b1 = min(b0 + 2, nb);
                        int sl = slot + min(b0 + (lane & 1), b1 - 1);
                        const uint32_t ph = sl >= a.stages ? phase ^ 1 : phase;
                        if (sl >= a.stages) sl -= a.stages;
                        if (!(ok = wait(&full[sl], ph))) break;
                        tc_fence_after();
                        if (elect_one()) {
                            sl = slot + b0 >= a.stages ? slot + b0 - a.stages : slot + b0;
                            for (int b = b0; b < b1; ++b) {
                                const uint32_t off = (uint32_t)sl * stage_bytes / 16;
                                if (b == 0) issue<NT, 0, 4>(tmem, col3, fresh, alo0 + off, ahi, blo0 + off, bhi);
                                else issue<NT, 0, 4>(tmem, col3, 0u, alo0 + off, ahi, blo0 + off, bhi);
                                if (++sl == a.stages) sl = 0;
                            }
                            if (b1 == nb) mma_commit(&gfull[ch & 1]);
                        }
                        __syncwarp();
                    }
                    if (!ok) break;
                    if (!(ok = wait(&gempty[2], (ch & 1) ^ 1))) break;
                    tc_fence_after();
                    if (elect_one()) {
                        int sl = slot;
                        for (int b = 0; b < nb; ++b) {
                            const uint32_t off = (uint32_t)sl * stage_bytes / 16;
                            if (b == 0) issue<NT, 4, 7>(tmem, 0u, fresh, alo0 + off, ahi, blo0 + off, bhi);
                            else issue<NT, 4, 7>(tmem, 0u, 0u, alo0 + off, ahi, blo0 + off, bhi);
                            mma_commit(&empty[sl]);
                            if (++sl == a.stages) sl = 0;
                        }
                        mma_commit(&gfull[2]);
                    }
                    __syncwarp();
                    slot += nb;
                    if (slot >= a.stages) {
                        slot -= a.stages;
                        phase ^= 1;
                    }
                }
            }
            if (elect_one()) mma_commit(mma_done);
            __syncwarp();
            volatile int no_abort = 0;
            mbar_wait(mma_done, 0, &no_abort, err, 2u, 100000000ull);
        } else {
            // ------------------------------------------------------------ sums of magnitudes
            Pieces<GemmArgs> pc(a);
            int tile, c0, c1;
            while (pc.next(a, &tile, &c0, &c1)) {
                if (c0 != 0) continue;             // the tile's first piece looks at all of the reduction
                const int2 at = tile_at(a, tile);
                list_small_sums<NT>(a, at.x, at.y, warp - 2, lane);
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, a.tmem_cols);
}

// The partial tiles of a split reduction, added in the order of the groups.
// (Of a listed, symmetric product the entries above the diagonal, both ways.)
// MANY: kManyParts and more (one tile spread over all SMs: 152, 27 us one after
// the other): eight warps take an eighth each, their sums are added in order
// (12.5 us with the leftovers of an unrolled loop, 7.7 us by sum_parts).
constexpr int kManyParts = 24;
template <bool MANY>
__global__ void __launch_bounds__(256) part_sum_kernel(const __grid_constant__ GemmArgs a, int NT, int64_t Q, int64_t G,
                                                       double* __restrict__ C, const double* __restrict__ rscale,
                                                       const double* __restrict__ cscale) {
    pdl_wait();
    pdl_trigger();
    const int tile = blockIdx.x;
    const int2 at = tile_at(a, tile);
    const int64_t u = (int64_t)(tile / a.group) * a.chunks;
    const int64_t p0 = group_of_chunk(u, Q, G), p1 = group_of_chunk(u + a.chunks - 1, Q, G);
    const double* part = a.C + (int64_t)tile * (128 * NT);
    const int64_t step = (int64_t)a.group * (128 * NT);
    auto put = [&](int e, double s) {
        const int64_t row = at.x * 128 + (e & 127), col = (int64_t)at.y * NT + (e >> 7);
        if (row >= a.M || col >= a.N || (a.listed && row > col)) return;
        if (rscale) s *= __ldg(rscale + row);
        if (cscale) s *= __ldg(cscale + col);
        C[row * a.cr + col * a.cc] = s;
        if (a.listed) C[col * a.cr + row * a.cc] = s;
    };
    if (!MANY) {
        for (int e = blockIdx.y * 256 + threadIdx.x; e < 128 * NT; e += 256 * gridDim.y) {
            put(e, sum_parts<4>(0.0, part + e, step, p0, p1 + 1));   // eight: 7.6 -> 10 us at 17 parts
        }
        return;
    }
    __shared__ double sm[8][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t np = p1 - p0 + 1, q0 = p0 + np * w / 8, q1 = p0 + np * (w + 1) / 8;
    for (int e0 = blockIdx.y * 32; e0 < 128 * NT; e0 += 32 * gridDim.y) {
        double s = sum_parts<8>(0.0, part + e0 + lane, step, q0, q1);
        __syncthreads();
        sm[w][lane] = s;
        __syncthreads();
        if (w == 0) {
            s = sm[0][lane];
#pragma unroll
            for (int i = 1; i < 8; ++i) s += sm[i][lane];
            put(e0 + lane, s);
        }
    }
}

// ---------------------------------------------------------------- repair
// Of the listed blocks the entries whose sums of magnitudes stay below the limit
// over all of the reduction, by binary64 FMAs, whose rate (two a clock on an SM) is
// the bound where there are many.  A warp takes 16 x 8 entries.
//  * Reductions from kLongK on: 8 x 4 entries at a time with the lanes along the
//    reduction, or where there are few one after the other.
//  * Shorter ones: four entries a lane.
struct RepairArgs {
    View64 A, B;
    const int2* fix;
    const int* nfix;
    int64_t M, N, K;
    double* C;
    int64_t cr, cc;
    const double* rscale;
    const double* cscale;
    int sym;                  // C symmetric, the entries above the diagonal are formed
    int groups;               // of 8 columns in a block
    const unsigned char* ia;  // images and kinds of rows
    const unsigned char* ib;
    const unsigned char* ka;
    const unsigned char* kb;
    int64_t a_block, b_block;
    int kblocks;
};
constexpr int kLongK = 96, kFew = 4;

__device__ __forceinline__ void put_entry(const RepairArgs& a, int64_t row, int64_t col, double s) {
    if (a.rscale) s *= __ldg(a.rscale + row);
    if (a.cscale) s *= __ldg(a.cscale + col);
    a.C[row * a.cr + col * a.cc] = s;
    if (a.sym) a.C[col * a.cr + row * a.cc] = s;
}

// One entry: lanes along the reduction, eight loads of either operand in flight.
__device__ __forceinline__ void repair_dot(const RepairArgs& a, int64_t row, int64_t col, int lane) {
    double s = 0.0;
    for (int64_t k0 = 0; k0 < a.K; k0 += 256) {
        double x[8], y[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int64_t k = k0 + 32 * u + lane;
            x[u] = k < a.K ? a.A.at(row, k) : 0.0;
            y[u] = k < a.K ? a.B.at(col, k) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) s = fma(x[u], y[u], s);
    }
#pragma unroll
    for (int o = 16; o > 0; o /= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) put_entry(a, row, col, s);
}

// Rows r0 ... r0 + 7 and columns c0, c0 + 2, c0 + 4, c0 + 6, bit 4 row + column / 2 of `mask`.
__device__ __forceinline__ void repair_word(const RepairArgs& a, int64_t r0, int64_t c0, uint32_t mask, int lane) {
    // an entry that is not listed may lie past the edge: the last listed one's row or column instead
    uint32_t cols = mask | mask >> 16;
    cols = (cols | cols >> 8 | cols >> 4 | cols >> 12) & 15u;
    const int rmax = (31 - __clz((int)mask)) / 4, cmax = 31 - __clz((int)cols);
    double acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.0;
    for (int64_t k = lane; k < a.K; k += 32) {
        double x[8], y[4];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = a.A.at(r0 + min(i, rmax), k);
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = a.B.at(c0 + 2 * min(j, cmax), k);
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = fma(x[i / 4], y[i % 4], acc[i]);
    }
    // the lanes' sums: lane l ends with entry l's
#pragma unroll
    for (int o = 16; o > 0; o /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const double mine = up ? acc[i + o] : acc[i], other = up ? acc[i] : acc[i + o];
            acc[i] = mine + __shfl_xor_sync(0xffffffffu, other, o);
        }
    }
    if ((mask >> lane) & 1) put_entry(a, r0 + lane / 4, c0 + 2 * (lane & 3), acc[0]);
}

// What a sum of first digits starts from, so that kMinSum is the limit for all: a
// row of zeros makes zeros, unless the other holds an infinity or a NaN.
__device__ __forceinline__ float first_sum(int ka, int kb) {
    if ((ka == kZeroRow && kb != kHardRow) || (kb == kZeroRow && ka != kHardRow)) return kMinSum;
    return ka == kDeepRow && kb == kDeepRow ? 0.0f : kMinSum - kMinShort;
}

// The entries of rows r0 ... r0 + 15 and columns c0 ... c0 + 7 that stay below the
// limit: bit `lane` of m[2 h + i] is row r0 + 8 h + lane / 4, column c0 + 2 (lane %
// 4) + i.  Eight blocks' digits in flight.
__device__ __forceinline__ void small_sums(const RepairArgs& a, int64_t r0, int64_t c0, int lane, uint32_t (&m)[4]) {
    const unsigned char* pa = a.ia + (r0 >> 3) * kGroupBytes;
    const unsigned char* pb = a.ib + (c0 >> 3) * kGroupBytes;
    float acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t r = r0 + 8 * (i >> 1) + lane / 4, c = c0 + 2 * (lane & 3) + (i & 1);
        const bool in = r < a.M && c < a.N && !(a.sym && r > c);
        acc[i] = in ? first_sum(a.ka[r], a.kb[c]) : kMinSum;
    }
    auto least = [&]() { return fminf(fminf(acc[0], acc[1]), fminf(acc[2], acc[3])); };
    bool done = false;
    for (int kb = 0; kb < a.kblocks && !done; kb += 8) {
        uint32_t x[8][4], y[8][2];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool in = kb + u < a.kblocks;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                x[u][i] = in ? first_digits(pa + (kb + u) * a.a_block + (i & 1) * kGroupBytes, i >> 1, lane) : 0u;
#pragma unroll
            for (int i = 0; i < 2; ++i) y[u][i] = in ? first_digits(pb + (kb + u) * a.b_block, i, lane) : 0u;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) mma_16x8(acc, x[u], y[u], acc[0], acc[1], acc[2], acc[3]);
        done = __all_sync(0xffffffffu, least() >= kMinSum) != 0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = __ballot_sync(0xffffffffu, !(acc[i] >= kMinSum));
}

__global__ void __launch_bounds__(256, 2) repair_kernel(const __grid_constant__ RepairArgs a) {
    pdl_wait();
    pdl_trigger();
    const int64_t units = (int64_t)*a.nfix * a.groups;
    if (units == 0) return;
    const int lane = threadIdx.x & 31;
    const int64_t w0 = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5), warps = (int64_t)gridDim.x * 8;
    // Few units with a long reduction: several warps each, with a word or with their
    // share of the entries.
    const int share = a.K < kLongK || units * 4 > warps ? 1 : units * 8 > warps ? 4 : units * 32 > warps ? 8 : 32;
    for (int64_t u = w0; u < units * share; u += warps) {
        const int mine = (int)(u % share), j = (int)(u / share % a.groups);
        const int2 f = a.fix[u / share / a.groups];
        const int64_t r0 = f.x, c0 = f.y + 8 * j;
        if (c0 >= a.N) continue;
        uint32_t m[4];
        small_sums(a, r0, c0, lane, m);
        if (!(m[0] | m[1] | m[2] | m[3])) continue;
        if (a.K >= kLongK) {
            int e = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (share == 4 && mine != i) continue;
                const int64_t rw = r0 + 8 * (i >> 1), cw = c0 + (i & 1);
                if (share <= 4 && __popc(m[i]) > kFew) {
                    repair_word(a, rw, cw, m[i], lane);
                } else {
                    for (uint32_t w = m[i]; w; w &= w - 1, ++e) {
                        const int bit = __ffs((int)w) - 1;
                        if (share <= 4 || e % share == mine) repair_dot(a, rw + bit / 4, cw + 2 * (bit & 3), lane);
                    }
                }
            }
            continue;
        }
        bool on[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) on[i] = (m[i] >> lane) & 1;
        const bool top = on[0] || on[1], low = on[2] || on[3], left = on[0] || on[2], right = on[1] || on[3];
        if (top || low) {
            // an entry that is not listed may lie past the edge: a listed one's row or column instead
            const int64_t r = r0 + lane / 4, c = c0 + 2 * (lane & 3);
            const int64_t ra = top ? r : r + 8, rb = low ? r + 8 : r, ca = left ? c : c + 1, cb = right ? c + 1 : c;
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
            for (int64_t k = 0; k < a.K; ++k) {
                const double x0 = a.A.at(ra, k), x1 = a.A.at(rb, k), y0 = a.B.at(ca, k), y1 = a.B.at(cb, k);
                acc[0] = fma(x0, y0, acc[0]);
                acc[1] = fma(x0, y1, acc[1]);
                acc[2] = fma(x1, y0, acc[2]);
                acc[3] = fma(x1, y1, acc[3]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (on[i]) put_entry(a, r + 8 * (i >> 1), c + (i & 1), acc[i]);
        }
        __syncwarp();
    }
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

int stat_splits(int64_t rows, int64_t K) {
    // eight CTAs a SM, at least 256 columns each
    const int64_t groups = (rows + 31) / 32;
    int64_t z = (8 * (int64_t)sm_count() + groups - 1) / groups;
    z = std::min<int64_t>(z, (K + 255) / 256);
    return (int)std::max<int64_t>(1, std::min<int64_t>(z, kStatSplits));
}

template <int NT>
lrc_status launch_product(const GemmArgs& a, const CUtensorMap& tm, int64_t grid, size_t smem, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(product_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(e, "split product_kernel smem attribute");
    e = launch_pdl(product_kernel<NT>, dim3((unsigned)grid), dim3(kThreads), smem, s, a, tm);
    if (e != cudaSuccess) return cuda_fail(e, "split product_kernel launch");
    return after_launch("split product_kernel");
}

}  // namespace

size_t operand_bytes(int64_t rows, int64_t K) {
    const int64_t ir = image_rows(rows);
    return up256((size_t)(ir / 8) * image_blocks(K) * kGroupBytes + kTailBytes) + up256((size_t)ir * 4) +
           up256((size_t)ir) + up256((size_t)rows * (K > kOwnStatsK ? kStatSplits : 0) * 4);
}

void operand_carve(Operand64* o, unsigned char* ws) {
    const int64_t ir = image_rows(o->rows);
    o->img = ws;
    ws += up256((size_t)(ir / 8) * image_blocks(o->K) * kGroupBytes + kTailBytes);
    o->exps = reinterpret_cast<int*>(ws);
    ws += up256((size_t)ir * 4);
    o->kind = ws;
    ws += up256((size_t)ir);
    o->stats = reinterpret_cast<int*>(ws);
}

lrc_status slice(const Operand64* const* ops, int count, int* clear, int nclear, cudaStream_t s) {
    Jobs st{}, sl{};
    st.clear = clear;
    st.nclear = nclear;
    int64_t bs = 0, bl = 0;
    for (int i = 0; i < count; ++i) {
        const Operand64& o = *ops[i];
        Job j{};
        j.v = View64{o.src};
        j.rows = o.rows;
        j.K = o.K;
        j.img_rows = image_rows(o.rows);
        j.kblocks = image_blocks(o.K);
        j.vec = o.src.cs == 1 && o.src.rs % 2 == 0 && aligned16(o.src.p);
        j.stats = o.stats;
        j.img = o.img;
        j.exps = o.exps;
        j.kind = o.kind;
        if (o.K > kOwnStatsK) {
            const int z = stat_splits(o.rows, o.K);
            j.kchunk = ((o.K + z - 1) / z + 31) / 32 * 32;
            j.splits = (int)((o.K + j.kchunk - 1) / j.kchunk);
            j.b0 = bs;
            bs += (o.rows + 31) / 32 * j.splits;
            st.j[st.n++] = j;
            j.kchunk = 256;
        } else {
            j.kchunk = j.kblocks * kKB;
        }
        j.kparts = (int)((j.kblocks * kKB + j.kchunk - 1) / j.kchunk);
        j.b0 = bl;
        bl += (j.img_rows + 31) / 32 * j.kparts;
        sl.j[sl.n++] = j;
    }
    if (bs > 0x7fffffff || bl > 0x7fffffff) {
        set_error("split product: operand too large");
        return LRC_ERR_UNSUPPORTED;
    }
    lrc_status r;
    cudaError_t e;
    if (st.n == 0) {
        if (nclear > 0 && (e = cudaMemsetAsync(clear, 0, nclear * sizeof(int), s)) != cudaSuccess)
            return cuda_fail(e, "cudaMemsetAsync (counters)");
    } else {
        e = launch_pdl(row_stats_kernel, dim3((unsigned)bs), dim3(256), 0, s, st);
        if (e != cudaSuccess) return cuda_fail(e, "row_stats_kernel launch");
        if ((r = after_launch("row_stats_kernel")) != LRC_OK) return r;
    }
    e = launch_pdl(slice_kernel, dim3((unsigned)bl), dim3(256), 0, s, sl);
    if (e != cudaSuccess) return cuda_fail(e, "slice_kernel launch");
    return after_launch("slice_kernel");
}

namespace {

int64_t n_tiles(int64_t rows) { return (rows + n_tile(rows) - 1) / n_tile(rows); }

// Tiles of a product with M rows on the first side; the side whose tiles waste
// less goes there.
int64_t tiles_of(int64_t M, int64_t N) { return (M + 127) / 128 * n_tiles(N); }

}  // namespace

size_t part_bytes(int64_t M, int64_t N) {
    if (tiles_of(N, M) < tiles_of(M, N)) std::swap(M, N);
    return up256((size_t)(tiles_of(M, N) + sm_count()) * 128 * n_tile(N) * 8);
}

int product_tile(int64_t M, int64_t N) { return tiles_of(N, M) < tiles_of(M, N) ? n_tile(M) : n_tile(N); }

size_t fix_bytes(int64_t M, int64_t N) {
    if (tiles_of(N, M) < tiles_of(M, N)) std::swap(M, N);
    return up256((size_t)((M + 15) / 16) * (size_t)(2 * n_tiles(N)) * sizeof(int2));
}

namespace {

lrc_status run_product(const Operand64& A0, const Operand64& B0, const Out64& out0, bool split, double* part,
                       const Fix& fix, bool sym, cudaStream_t s) {
    const bool swap = tiles_of(B0.rows, A0.rows) < tiles_of(A0.rows, B0.rows);
    const Operand64& A = swap ? B0 : A0;
    const Operand64& B = swap ? A0 : B0;
    Out64 out = out0;
    if (swap) {
        std::swap(out.cr, out.cc);
        std::swap(out.rscale, out.cscale);
    }
    const int NT = n_tile(B.rows);
    GemmArgs a{};
    a.A = A.img;
    a.B = B.img;
    a.ea = A.exps;
    a.eb = B.exps;
    a.C = split ? part : out.C;
    a.fix = fix.list;
    a.nfix = fix.count;
    a.cr = out.cr;
    a.cc = out.cc;
    a.M = A.rows;
    a.N = B.rows;
    int64_t tiles = tiles_of(A.rows, B.rows);
    if (tiles > 0x3fffffff || A.K > kMaxK) {
        set_error("split product too large (%lld tiles, reduction of %lld)", (long long)tiles, (long long)A.K);
        return LRC_ERR_UNSUPPORTED;
    }
    a.ntiles = (int)n_tiles(B.rows);
    if (sym && tiles <= 2 * kMaxListed) {
        int n = 0;
        for (int mt = 0; mt < (int)(tiles / a.ntiles); ++mt)
            for (int nt = 0; nt < a.ntiles; ++nt)
                if ((nt + 1) * NT > mt * 128) {
                    if (n < kMaxListed) a.list[n] = (uint16_t)(mt << 8 | nt);
                    ++n;
                }
        if (n <= kMaxListed) {
            a.listed = n;
            tiles = n;
        }
    }
    a.tiles = (int)tiles;
    a.kblocks = (int)image_blocks(A.K);
    a.chunks = (a.kblocks + kChunkBlocks - 1) / kChunkBlocks;
    a.split = split;
    a.a_block = image_rows(A.rows) / 8 * kGroupBytes;
    a.b_block = image_rows(B.rows) / 8 * kGroupBytes;
    a.a_bytes = 128 / 8 * kGroupBytes;
    a.b_bytes = (uint32_t)(NT / 8 * kGroupBytes);
    CUtensorMap tm{};
    a.tma = !split && out.cc == 1 && out.cr % 2 == 0 && aligned16(out.C);
    lrc_status st;
    if (a.tma) {
        const bool wide = NT % 32 == 0;      // columns a warp stores at a time: 8, else 4
        st = wide ? encode_map_2d_sw64(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, out.C, B.rows, A.rows, out.cr * 8, 8, 32,
                                       "split product output")
                  : encode_map_2d(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, out.C, B.rows, A.rows, out.cr * 8, 4, 32, false,
                                  "split product output");
        if (st != LRC_OK) return st;
    }
    // (a chunk's blocks are all in the ring at once: at least kChunkBlocks stages)
    const size_t staging = !split && out.cc == 1 ? (size_t)kEpiWarps * kStageBytes : 0;
    a.stages = (int)std::min<int64_t>(8, (int64_t)(227 * 1024 - kCtrlBytes - staging) / (a.a_bytes + a.b_bytes));
    uint32_t cols = 32;
    while (cols < (uint32_t)(8 * NT)) cols *= 2;
    a.tmem_cols = cols;
    const int64_t sms = sm_count();
    // groups of one CTA per tile of B while that leaves at least eight groups
    a.group = split && !a.listed && (int64_t)a.ntiles * 8 <= sms ? a.ntiles : 1;
    const int64_t Q = tiles / a.group * a.chunks;
    const int64_t groups = std::min<int64_t>(Q, sms / a.group);
    const int64_t grid = split ? groups * a.group : std::min<int64_t>(tiles, sms);
    const size_t smem = kCtrlBytes + (size_t)a.stages * (a.a_bytes + a.b_bytes) + staging;
    switch (NT) {
        case 16: st = launch_product<16>(a, tm, grid, smem, s); break;
        case 32: st = launch_product<32>(a, tm, grid, smem, s); break;
        case 48: st = launch_product<48>(a, tm, grid, smem, s); break;
        default: st = launch_product<64>(a, tm, grid, smem, s); break;
    }
    if (st != LRC_OK) return st;
    cudaError_t e;
    if (split) {
        const bool many = groups / (tiles / a.group) >= kManyParts;
        const int64_t most = 128 * NT / (many ? 32 : 256), want = (many ? 8 : 4) * sms / tiles;
        const unsigned gy = (unsigned)std::max<int64_t>(1, std::min(most, want));
        e = launch_pdl(many ? part_sum_kernel<true> : part_sum_kernel<false>, dim3((unsigned)tiles, gy), dim3(256), 0,
                       s, a, NT, Q, groups, out.C, out.rscale, out.cscale);
        if (e != cudaSuccess) return cuda_fail(e, "part_sum_kernel launch");
        if ((st = after_launch("part_sum_kernel")) != LRC_OK) return st;
    }
    const RepairArgs r{View64{A.src}, View64{B.src}, fix.list, fix.count, A.rows, B.rows, A.K, out.C, out.cr, out.cc,
                       out.rscale, out.cscale, a.listed ? 1 : 0, NT / 16, A.img, B.img, A.kind, B.kind,
                       a.a_block, a.b_block, a.kblocks};
    e = launch_pdl(repair_kernel, dim3((unsigned)(2 * sms)), dim3(256), 0, s, r);
    if (e != cudaSuccess) return cuda_fail(e, "repair_kernel launch");
    return after_launch("repair_kernel");
}

}  // namespace

lrc_status product(const Operand64& A, const Operand64& B, const Out64& out, bool split, double* part, const Fix& fix,
                   cudaStream_t s) {
    return run_product(A, B, out, split, part, fix, false, s);
}

lrc_status gram(const Operand64& A, double* C, int64_t ldc, double* part, const Fix& fix, cudaStream_t s) {
    return run_product(A, A, Out64{C, ldc, 1, nullptr, nullptr}, true, part, fix, true, s);
}

}  // namespace sg

uint32_t take_split_error() {
    unsigned int v = 0;
    if (cudaMemcpyFromSymbol(&v, sg::g_err_split, sizeof v) != cudaSuccess) return 0xffffffffu;
    if (v) {
        const unsigned int z = 0;
        cudaMemcpyToSymbol(sg::g_err_split, &z, sizeof z);
    }
    return v;
}

}  // namespace lrc
