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
//     are below 2^-62 and are left out (28 products of 49).
//   * every 64 terms (`period`: less often where the bound allows) the
//     accumulators are drained into two 64-bit integers per entry, and the
//     whole sum is rounded to binary64 once.
//
// So the result is as close as the best rounded one for rows whose entries
// lie within about 2^-9 of each other's scale, and the error never exceeds
// about 2^-61 of (largest of row i)(largest of row j) per term.  Rows that
// this does not describe well -- their entries lie on average more than
// 2^-kMaxGap below the largest, or they hold an infinity, a NaN or a largest
// entry outside 2^-480 ... 2^495 -- get zero digits and are
// recomputed by a kernel of binary64 FMAs (`repair`).
//
// Kernels: row statistics (row_stats_kernel), digits (slice_kernel, which
// writes them as images that either side of a product loads by bulk copies), the product (product_kernel,
// persistent, one CTA a SM), the ordered sum of split reductions
// (part_sum_kernel) and the repair (repair_kernel).
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
constexpr int kMaxGap = 12;            // mean distance (in bits) of a row's entries below its largest
constexpr int kNonFinite = 1 << 20;    // marks a row with an infinity or NaN in its statistics
// Biased exponents of a row's largest entry that digits carry: with both rows
// inside, every result is zero or a normal number (round96).
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
// Per row: the largest biased exponent, the sum of the exponents of the
// nonzero entries and their number.
struct RowStat {
    int mx = -(1 << 20), sum = 0, cnt = 0;
    __device__ __forceinline__ void add(double x, int shift) {
        const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu, e = h >> 20;
        int v = (int)e + shift, one = 1;
        if (e - 1u >= 0x7feu) {            // zero, subnormal, infinity or NaN
            one = (h | (uint32_t)__double2loint(x)) != 0 ? 1 : 0;
            v = one ? biased_exp(((uint64_t)h << 32) | (uint32_t)__double2loint(x)) + shift : -(1 << 20);
        }
        mx = max(mx, v);
        sum += one && v < kNonFinite / 2 ? v : 0;
        cnt += one;
    }
    __device__ __forceinline__ void merge(int4 o) {
        mx = max(mx, o.x);
        sum += o.y;
        cnt += o.z;
    }
};

// What the kernels below take of an operand, and its share of the blocks.
struct Job {
    View64 v;
    int64_t rows, K, img_rows, kblocks;
    int64_t b0;              // first block
    int64_t kchunk;          // columns a block takes
    int kparts, splits, vec;
    int4* stats;             // splits > 0: statistics per slice of K; else slice_kernel takes its own
    unsigned char* img;
    int* exps;
    int* hard;
};
struct Jobs {
    Job j[kMaxOps];
    int n;
    int* clear[kMaxOps];     // row lists to empty
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
__device__ __forceinline__ RowStat block_stats(const View64& v, int64_t r0, int64_t rows, int64_t k0, int64_t k1,
                                               bool vec, int4 (&sm)[8][32]) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto shift = [&](int64_t k) { return SCALED ? v.shift(k) : 0; };
    if (v.s.cs == 1) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t r = r0 + warp + 8 * q;
            RowStat a;
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
                            a.add(x[u].x, shift(k + 64 * u));
                            a.add(x[u].y, shift(k + 64 * u + 1));
                        }
                    }
                }
                for (; k < k1; k += 64) {
                    a.add(v.at(r, k), shift(k));
                    if (k + 1 < k1) a.add(v.at(r, k + 1), shift(k + 1));
                }
            }
            a.mx = __reduce_max_sync(0xffffffffu, a.mx);
            a.sum = __reduce_add_sync(0xffffffffu, a.sum);
            a.cnt = __reduce_add_sync(0xffffffffu, a.cnt);
            if (lane == 0) sm[0][warp + 8 * q] = make_int4(a.mx, a.sum, a.cnt, 0);
        }
    } else {
        const int64_t r = r0 + lane;
        RowStat a;
        if (r < rows) {
            int64_t k = k0 + warp;
            for (; k + 24 < k1; k += 32) {
                double x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = v.at(r, k + 8 * u);
#pragma unroll
                for (int u = 0; u < 4; ++u) a.add(x[u], shift(k + 8 * u));
            }
            for (; k < k1; k += 8) a.add(v.at(r, k), shift(k));
        }
        sm[warp][lane] = make_int4(a.mx, a.sum, a.cnt, 0);
    }
    __syncthreads();
    RowStat t;
    if (warp == 0) {
        t.merge(sm[0][lane]);
        if (v.s.cs != 1) {
#pragma unroll
            for (int w = 1; w < 8; ++w) t.merge(sm[w][lane]);
        }
    }
    return t;
}

__global__ void __launch_bounds__(256) row_stats_kernel(const __grid_constant__ Jobs js) {
    __shared__ int4 sm[8][32];
    pdl_wait();
    pdl_trigger();
    const Job& o = job_of(js, blockIdx.x);
    const int64_t lb = (int64_t)blockIdx.x - o.b0, rg = lb / o.splits, z = lb - rg * o.splits;
    const int64_t r0 = rg * 32, k0 = z * o.kchunk;
    if (blockIdx.x == 0 && threadIdx.x < kMaxOps && js.clear[threadIdx.x]) *js.clear[threadIdx.x] = 0;
    const int64_t k1 = min(o.K, k0 + o.kchunk);
    const RowStat a = o.v.s.scale ? block_stats<true>(o.v, r0, o.rows, k0, k1, o.vec != 0, sm)
                                  : block_stats<false>(o.v, r0, o.rows, k0, k1, o.vec != 0, sm);
    if (threadIdx.x < 32 && r0 + threadIdx.x < o.rows)
        o.stats[z * o.rows + r0 + threadIdx.x] = make_int4(a.mx, a.sum, a.cnt, 0);
}

// ---------------------------------------------------------------- digits
// The seven digits of eight values as bfloat16: w[p][q] holds digits
// p of values 2q (low half) and 2q + 1.  em: biased exponent of the row's
// largest entry.  The value is rounded to a multiple of 2^-61 of 2^(em -
// 1022), the power of two above it, and the digits are those of that integer
// plus 256 at every place but the first, minus 256 again: a number read with
// digits in [-256, 255].
__device__ __forceinline__ void digits8(const double (&x)[8], const int (&sh)[8], int em, uint32_t (&w)[kParts64][4]) {
    constexpr uint64_t kBias = 256ull * (1ull + (1ull << 9) + (1ull << 18) + (1ull << 27) + (1ull << 36) + (1ull << 45));
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
__global__ void __launch_bounds__(256) slice_kernel(const __grid_constant__ Jobs js) {
    __shared__ int4 sm[8][32];
    __shared__ int s_em[32];
    pdl_wait();
    pdl_trigger();
    const Job& o = job_of(js, blockIdx.x);
    const View64 v = o.v;
    const int64_t rows = o.rows, K = o.K;
    const int64_t lb = (int64_t)blockIdx.x - o.b0, rg = lb / o.kparts, kp = lb - rg * o.kparts;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t r0 = rg * 32;
    RowStat own;
    if (o.splits == 0) own = block_stats<true>(v, r0, rows, 0, K, o.vec != 0, sm);
    if (tid < 32) {
        const int64_t r = r0 + lane;
        int em = 1023;
        bool zero = true;
        if (r < rows) {
            int mx = own.mx;
            int64_t sum = own.sum, cnt = own.cnt;
            for (int z = 0; z < o.splits; ++z) {
                const int4 a = o.stats[(int64_t)z * rows + r];
                mx = max(mx, a.x);
                sum += a.y;
                cnt += a.z;
            }
            if (cnt > 0) {
                zero = mx < kMinExp || mx > kMaxExp || (int64_t)mx * cnt - sum > (int64_t)kMaxGap * cnt;
                if (!zero) em = mx;
                else if (kp == 0) o.hard[1 + atomicAdd(o.hard, 1)] = (int)r;
            }
        }
        s_em[lane] = zero ? -1 : em;
        if (kp == 0 && r < o.img_rows) o.exps[r] = em;
    }
    __syncthreads();
    const int64_t r = r0 + lane;
    if (r >= o.img_rows) return;
    const int em = s_em[lane];
    const size_t block_bytes = (size_t)(o.img_rows / 8) * kGroupBytes;
    unsigned char* row_base = o.img + (size_t)(r >> 3) * kGroupBytes + (r & 7) * 16;
    const int64_t o1 = min((kp + 1) * o.kchunk, o.kblocks * kKB) / 8;
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
        digits8(x, sh, em < 0 ? 1023 : em, w);
        unsigned char* dst = row_base + (size_t)(oc >> 1) * block_bytes + (size_t)(oc & 1) * 128;
#pragma unroll
        for (int i = 0; i < kParts64; ++i)
            *reinterpret_cast<uint4*>(dst + i * (8 * kKB * 2)) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
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
// Registers: the first four warps (producer, MMA issuer, two idle) hand some
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
                                                       const double* __restrict__ cscale, int* __restrict__ clear) {
    pdl_wait();
    pdl_trigger();
    if (clear && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *clear = 0;
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
// Rows listed as hard: their part of C by binary64 FMAs.  The binary64 pipe (two
// FMAs a clock on an SM) is the bound, as for the FMA kernels of the other paths;
// with every row listed (factors whose entries decay over many binades) a product
// should take what it takes there.  So the tile follows from how many there are:
// R x R entries a thread in tiles of 16 R, and for few entries (R = 0) tiles of
// 8 x 8 whose reduction is split over four threads.  With entries over 60 binades
// in both operands: apply 16384 x 8192, k = 128, b = 2048 11.3 ms (FMA kernels
// 11.2), 12287 x 16384, k = 272, b = 250 4.1 ms (4.2); 64 x 64 tiles alone
// took about 100 ms for results of 140 x 104 with a reduction of 71680.
struct RepairArgs {
    View64 A, B;
    const int* ha;
    const int* hb;
    int64_t M, N, K;
    double* C;
    int64_t cr, cc;
    const double* rscale;
    const double* cscale;
    int sym;                  // A and B are the same operand, C symmetric
};
constexpr int kRepairWords = 128 * 9;        // staged entries of an operand, with padding (the largest of all R)

template <int R>
__host__ __device__ constexpr int repair_tile() { return R == 0 ? 8 : 16 * R; }

__device__ __forceinline__ int64_t repair_tiles(int64_t na, int64_t nb, int64_t M, int64_t N, int T) {
    return (na + T - 1) / T * ((N + T - 1) / T) + (nb + T - 1) / T * ((M + T - 1) / T);
}

template <int R>
__device__ __forceinline__ void repair_body(const RepairArgs& a, int64_t na, int64_t nb, double* As, double* Bs) {
    constexpr int T = repair_tile<R>(), KS = 1024 / T, P = T + 1, E = R == 0 ? 1 : R, W = R == 0 ? 8 : 16;
    const int64_t ta = (na + T - 1) / T * ((a.N + T - 1) / T), tiles = repair_tiles(na, nb, a.M, a.N, T);
    const int tid = threadIdx.x;
    const int part = R == 0 ? tid / 64 : 0;                        // quarter of the reduction
    const int tx = tid % W, ty = R == 0 ? tid / 8 % 8 : tid / 16;
    const bool all = na == a.M;                                    // every row of A: in order, not by the list
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        // tile of C rows (first list entry or row) and columns
        const bool ga = t < ta;
        const int64_t u = ga ? t : t - ta;
        const int64_t other = ((ga ? a.N : a.M) + T - 1) / T;
        const int64_t l0 = u / other * T, o0 = (u % other) * T;
        const int64_t i0 = ga ? l0 : o0, j0 = ga ? o0 : l0;
        if (a.sym && all && i0 > j0) continue;                     // written with the tile above the diagonal
        const int64_t ni = ga ? na : a.M, nj = ga ? a.N : nb;
        auto row_of = [&](int i) {
            return i0 + i >= ni ? -1 : ga && !all ? __ldg(a.ha + 1 + i0 + i) : (int)(i0 + i);
        };
        auto col_of = [&](int j) { return j0 + j >= nj ? -1 : ga ? (int)(j0 + j) : __ldg(a.hb + 1 + j0 + j); };
        // a thread stages four entries of each operand, neighbours along k
        const int kk = tid % KS, x0 = tid / KS;
        constexpr int XS = 256 / KS > 0 ? 256 / KS : 1;
        static_assert(KS <= 256, "");
        int ri[4], cj[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            ri[q] = row_of(x0 + q * XS);
            cj[q] = col_of(x0 + q * XS);
        }
        double acc[E][E];
#pragma unroll
        for (int i = 0; i < E; ++i)
#pragma unroll
            for (int j = 0; j < E; ++j) acc[i][j] = 0.0;
        double va[4], vb[4];
        auto load = [&](int64_t k0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                va[q] = ri[q] >= 0 && k0 + kk < a.K ? a.A.at(ri[q], k0 + kk) : 0.0;
                vb[q] = cj[q] >= 0 && k0 + kk < a.K ? a.B.at(cj[q], k0 + kk) : 0.0;
            }
        };
        load(0);
        for (int64_t k0 = 0; k0 < a.K; k0 += KS) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                As[kk * P + x0 + q * XS] = va[q];
                Bs[kk * P + x0 + q * XS] = vb[q];
            }
            __syncthreads();
            if (k0 + KS < a.K) load(k0 + KS);                      // in flight over this slab's FMAs
            const int kn = (int)min((int64_t)KS, a.K - k0);
            const int kb = R == 0 ? part * (KS / 4) : 0, ke = R == 0 ? min(kn, kb + KS / 4) : kn;
#pragma unroll 4
            for (int k = kb; k < ke; ++k) {
                double x[E], y[E];
#pragma unroll
                for (int i = 0; i < E; ++i) x[i] = As[k * P + ty + W * i];
#pragma unroll
                for (int j = 0; j < E; ++j) y[j] = Bs[k * P + tx + W * j];
#pragma unroll
                for (int i = 0; i < E; ++i)
#pragma unroll
                    for (int j = 0; j < E; ++j) acc[i][j] = fma(x[i], y[j], acc[i][j]);
            }
            __syncthreads();
        }
        if (R == 0) {
            As[tid] = acc[0][0];
            __syncthreads();
            acc[0][0] = ((As[tid & 63] + As[64 + (tid & 63)]) + As[128 + (tid & 63)]) + As[192 + (tid & 63)];
            __syncthreads();
            if (part != 0) continue;
        }
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const int64_t row = row_of(ty + W * i);
            if (row < 0) continue;
#pragma unroll
            for (int j = 0; j < E; ++j) {
                const int64_t col = col_of(tx + W * j);
                if (col < 0) continue;
                double s = acc[i][j];
                if (a.rscale) s *= __ldg(a.rscale + row);
                if (a.cscale) s *= __ldg(a.cscale + col);
                a.C[row * a.cr + col * a.cc] = s;
                if (a.sym && all) a.C[col * a.cr + row * a.cc] = s;
            }
        }
    }
}

__global__ void __launch_bounds__(256, 2) repair_kernel(const __grid_constant__ RepairArgs a) {
    __shared__ double As[kRepairWords], Bs[kRepairWords];
    pdl_wait();
    pdl_trigger();
    const int64_t na = a.ha[0], nb = na == a.M ? 0 : a.hb[0];      // every row of A: all of C
    if (na + nb == 0) return;
    const int64_t grid = gridDim.x;
    if (repair_tiles(na, nb, a.M, a.N, 64) >= 2 * grid) repair_body<4>(a, na, nb, As, Bs);
    else if (repair_tiles(na, nb, a.M, a.N, 32) >= 2 * grid) repair_body<2>(a, na, nb, As, Bs);
    else if (repair_tiles(na, nb, a.M, a.N, 16) >= 4 * grid) repair_body<1>(a, na, nb, As, Bs);
    else repair_body<0>(a, na, nb, As, Bs);
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
           up256((size_t)rows * (K > kOwnStatsK ? kStatSplits : 0) * sizeof(int4)) + hard_bytes(rows);
}

void operand_carve(Operand64* o, unsigned char* ws) {
    const int64_t ir = image_rows(o->rows);
    o->img = ws;
    ws += up256((size_t)(ir / 8) * image_blocks(o->K) * kGroupBytes + kTailBytes);
    o->exps = reinterpret_cast<int*>(ws);
    ws += up256((size_t)ir * 4);
    o->stats = reinterpret_cast<int4*>(ws);
    ws += up256((size_t)o->rows * (o->K > kOwnStatsK ? kStatSplits : 0) * sizeof(int4));
    o->hard = reinterpret_cast<int*>(ws);
}

lrc_status slice(const Operand64* const* ops, int count, cudaStream_t s) {
    Jobs st{}, sl{};
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
        j.hard = o.hard;
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
        if (!o.cleared) st.clear[i] = o.hard;
    }
    if (bs > 0x7fffffff || bl > 0x7fffffff) {
        set_error("split product: operand too large");
        return LRC_ERR_UNSUPPORTED;
    }
    lrc_status r;
    cudaError_t e;
    if (st.n == 0) {
        for (int i = 0; i < count; ++i)
            if (st.clear[i] && (e = cudaMemsetAsync(st.clear[i], 0, sizeof(int), s)) != cudaSuccess)
                return cuda_fail(e, "cudaMemsetAsync (row list)");
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

namespace {

lrc_status run_product(const Operand64& A0, const Operand64& B0, const Out64& out0, bool split, double* part, bool sym,
                       cudaStream_t s) {
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
        const unsigned gy = (unsigned)std::max<int64_t>(1, std::min<int64_t>(128 * NT / (many ? 32 : 256), (many ? 8 : 4) * sms / tiles));
        e = launch_pdl(many ? part_sum_kernel<true> : part_sum_kernel<false>, dim3((unsigned)tiles, gy), dim3(256), 0,
                       s, a, NT, Q, groups, out.C, out.rscale, out.cscale, out.clear);
        if (e != cudaSuccess) return cuda_fail(e, "part_sum_kernel launch");
        if ((st = after_launch("part_sum_kernel")) != LRC_OK) return st;
    }
    const RepairArgs r{View64{A.src}, View64{B.src}, A.hard, B.hard, A.rows, B.rows, A.K, out.C, out.cr, out.cc,
                       out.rscale, out.cscale, sym ? 1 : 0};
    e = launch_pdl(repair_kernel, dim3((unsigned)(2 * sms)), dim3(256), 0, s, r);
    if (e != cudaSuccess) return cuda_fail(e, "repair_kernel launch");
    return after_launch("repair_kernel");
}

}  // namespace

lrc_status product(const Operand64& A, const Operand64& B, const Out64& out, bool split, double* part, cudaStream_t s) {
    return run_product(A, B, out, split, part, false, s);
}

lrc_status gram(const Operand64& A, double* C, int64_t ldc, double* part, cudaStream_t s) {
    return run_product(A, A, Out64{C, ldc, 1, nullptr, nullptr}, true, part, true, s);
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
