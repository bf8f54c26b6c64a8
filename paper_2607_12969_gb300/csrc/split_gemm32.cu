// split_gemm32.cu -- binary32 products C = A B^T on the tensor cores.
//
// The CUDA cores reach 42 to 47 TFLOP/s on these products; the tensor cores
// multiply bfloat16 numbers at 1700.  A binary32 value is the exact sum of three
// bfloat16 numbers, x = hi + mid + lo (each the nearest to what is left: mid at
// most 2^-8 of x, lo 2^-17), so of the nine products of parts the six largest,
//     hi hi + (hi mid + mid hi) + (mid mid + hi lo + lo hi),
// leave out at most 2^-24 of a term, binary32's own rounding of it, and 2^-26 as a
// rule.  Each value is split by itself: nothing depends on its neighbours.
//
// The tensor cores' binary32 accumulation cuts sums off (about 0.4 units of the
// last place a step of 16 terms, all in one direction), so hi hi runs for only
// 64 terms in its accumulator, which is then added to a running sum in
// registers with IEEE additions; the other five products, 2^-8 of the result,
// share an accumulator that is drained every 1024 terms.  Relative distance
// from binary64 of the apply (16384 x 8192, k = 136, b = 8192): 2.4e-7, with
// binary32 FMAs 6.5e-7.
//
// The parts are those of 2^24 x (2^48 comes off as an accumulator is added to the
// running sum): every binary32 number is a multiple of 2^-149, so its scaled parts
// are multiples of 2^-125, zero or normal bfloat16 numbers, and none is lost
// however small x is.  Entries are bounded, 2^40 on the first side and 2^32 on the
// second, so that no accumulator leaves binary32's range: a row with a larger one,
// an infinity or a NaN is recomputed with binary32 FMAs.  (Without such a bound two
// entries of 2^71 made hi hi infinite, hi mid the other infinity, and their sum a
// NaN.)
//
// Kernels: parts_kernel (the images), product32_kernel (persistent, one CTA a
// SM: 128 x up to 256 tiles), part_sum32_kernel (split reductions) and
// repair32_kernel.
#include <algorithm>

#include "split_gemm32.cuh"
#include "split_pieces.cuh"
#include "tc.cuh"

namespace lrc {
namespace sg32 {

namespace {

using namespace tc;

__device__ unsigned int g_err_split32;

// ---------------------------------------------------------------- parts
struct Job {
    const float* p;
    int64_t rs, cs, rows, K, img_rows, kblocks;
    int64_t b0;              // first block
    int kparts, vec;
    float limit;             // largest magnitude carried
    unsigned char* img;
    int* hard;
};
struct Jobs {
    Job j[3];
    int n;
};
constexpr int kJobCols = 256;      // columns a block takes
constexpr float kUp = 0x1p24f, kDown = 0x1p-48f;

// Largest entry carried on either side: 64 products of 2^48 times these stay
// below 2^126.
constexpr float kFirstLimit = 0x1p40f, kSecondLimit = 0x1p32f;

// The bits of the three parts of 2^24 x, each in the upper half of its word.
__device__ __forceinline__ void parts_of(float x0, uint32_t (&h)[kParts]) {
    const float x = __fmul_rn(x0, kUp);
    const float hi = __uint_as_float((uint32_t)to_bf16_bits(x) << 16);
    const float r1 = __fsub_rn(x, hi);
    const float mid = __uint_as_float((uint32_t)to_bf16_bits(r1) << 16);
    const float lo = __fsub_rn(r1, mid);
    h[0] = __float_as_uint(hi);
    h[1] = __float_as_uint(mid);
    h[2] = __float_as_uint(lo);            // eight bits: the truncation below is exact
}

// A CTA takes 32 rows and kJobCols columns; a lane is a row, so that a warp's
// 16-byte stores of one part are four runs of 128 bytes.
__global__ void __launch_bounds__(256) parts_kernel(const __grid_constant__ Jobs js) {
    pdl_wait();
    pdl_trigger();
    int ji = 0;
    while (ji + 1 < js.n && (int64_t)blockIdx.x >= js.j[ji + 1].b0) ++ji;
    const Job& o = js.j[ji];
    const int64_t lb = (int64_t)blockIdx.x - o.b0, rg = lb / o.kparts, kp = lb - rg * o.kparts;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r = rg * 32 + lane;
    const size_t block_bytes = (size_t)(o.img_rows / 8) * kGroupBytes;
    unsigned char* row_base = o.img + (size_t)(r >> 3) * kGroupBytes + (r & 7) * 16;
    const int64_t o1 = min((kp + 1) * (int64_t)kJobCols, o.kblocks * kKB) / 8;
    bool bad = false;
    for (int64_t oc = kp * (kJobCols / 8) + warp; oc < o1; oc += 8) {
        float x[8];
        const int64_t k0 = oc * 8;
        if (r >= o.rows) {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = 0.0f;
        } else if (o.vec && k0 + 8 <= o.K) {
            const float4* p = reinterpret_cast<const float4*>(o.p + r * o.rs + k0);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float4 d = __ldg(p + j);
                x[4 * j] = d.x;
                x[4 * j + 1] = d.y;
                x[4 * j + 2] = d.z;
                x[4 * j + 3] = d.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = k0 + j < o.K ? __ldg(o.p + r * o.rs + (k0 + j) * o.cs) : 0.0f;
        }
        uint32_t w[kParts][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t a[kParts], b[kParts];
            parts_of(x[2 * q], a);
            parts_of(x[2 * q + 1], b);
#pragma unroll
            for (int i = 0; i < kParts; ++i) w[i][q] = __byte_perm(a[i], b[i], 0x7632);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) bad |= !(fabsf(x[j]) <= o.limit);
        unsigned char* dst = row_base + (size_t)(oc >> 1) * block_bytes + (size_t)(oc & 1) * 128;
#pragma unroll
        for (int i = 0; i < kParts; ++i)
            *reinterpret_cast<uint4*>(dst + i * (8 * kKB * 2)) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
    }
    // each row joins the list once
    if (bad && atomicExch(o.hard + 1 + o.rows + r, 1) == 0) o.hard[1 + atomicAdd(o.hard, 1)] = (int)r;
}

// ---------------------------------------------------------------- product
struct GemmArgs {
    const unsigned char* A;
    const unsigned char* B;
    float* C;                // split: partial tiles [slot][column][128 rows]
    int64_t ldc, M, N;
    int ntiles, tiles;       // tiles of B; all tiles
    int chunks;              // 64-column chunks of the reduction
    int kblocks;             // 16-column blocks
    int split, group, stages, tma, NT;
    int64_t a_block, b_block;    // bytes of a block of either image
    uint32_t a_bytes, b_bytes;   // of a tile's part of it
    uint32_t tmem_cols;
};

constexpr int kEpiWarps = 16;
constexpr int kThreads = 32 * (4 + kEpiWarps);
constexpr int kChunkBlocks = 64 / kKB;
constexpr int kLowPeriod = 16;             // chunks between drains of the lower products
constexpr int kMaxCols = kNTMax / 4;       // columns a thread sums
constexpr uint32_t kCtrlBytes = 1024;
// The output leaves through shared memory, 32 x 32 a warp at a time: by TMA
// (128-byte rows in the 128-byte swizzle), or where a row's pitch does not allow
// that by runs of 128 bytes.  Stores of 32 bytes a lane straight from the
// registers filled the load/store unit: 236 us for 537 MB.
constexpr int kStagePitch = 33, kStageBytes = 5 * 1024;

__global__ void __launch_bounds__(kThreads, 1) product32_kernel(const __grid_constant__ GemmArgs a,
                                                                const __grid_constant__ CUtensorMap tm_c) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);
    uint64_t* empty = full + 8;
    uint64_t* gfull = empty + 8;        // accumulators complete: hi hi, the rest
    uint64_t* gempty = gfull + 2;       // ... drained
    uint64_t* mma_done = gempty + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
    volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
    unsigned char* ring = smem + kCtrlBytes;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t stage_bytes = a.a_bytes + a.b_bytes;
    unsigned int* err = &g_err_split32;
    const int NT = a.NT;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
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
        // ------------------------------------------------------------ epilogue
        const int g = warp & 3, quarter = (warp - 4) >> 2;      // of the lanes, of the columns
        const int hc = NT / 4;
        const uint32_t tbase = tmem + ((uint32_t)(g * 32) << 16) + quarter * hc;
        const int r = g * 32 + lane;
        float* stage = reinterpret_cast<float*>(ring + (size_t)a.stages * stage_bytes + (size_t)(warp - 4) * kStageBytes);
        sg::Pieces<GemmArgs> pc(a);
        int tile, c0, c1;
        int ch = 0, lo = 0;
        bool ok = true;
        // one warp polls the mbarrier, the others sleep at the named barrier
        auto epi_wait = [&](uint64_t* bar, uint32_t parity) {
            if (warp == 4) mbar_wait(bar, parity, abort, err, 4u);
            named_bar_sync(1, 32 * kEpiWarps);
            return *abort == 0;
        };
        while (ok && pc.next(a, &tile, &c0, &c1)) {
            float sum[kMaxCols];
#pragma unroll
            for (int j = 0; j < kMaxCols; ++j) sum[j] = 0.0f;
            // adds the thread's columns of an accumulator (past a quarter's end
            // another's, which are never stored)
            auto drain = [&](uint32_t taddr) {
#pragma unroll
                for (int j0 = 0; j0 < kMaxCols; j0 += 16) {
                    if (j0 < hc) {
                        uint32_t u[8], v[8];
                        tmem_ld8(taddr + j0, u);
                        tmem_ld8(taddr + j0 + 8, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            sum[j0 + j] = __fmaf_rn(__uint_as_float(u[j]), kDown, sum[j0 + j]);
                            sum[j0 + 8 + j] = __fmaf_rn(__uint_as_float(v[j]), kDown, sum[j0 + 8 + j]);
                        }
                    }
                }
            };
            for (int c = c0; c < c1; ++c, ++ch) {
                if (!(ok = epi_wait(&gfull[0], ch & 1))) break;
                tc_fence_after();
                drain(tbase);
                tc_fence_before();
                mbar_arrive(&gempty[0]);
                if (c + 1 == c1 || (c - c0 + 1) % kLowPeriod == 0) {
                    if (!(ok = epi_wait(&gfull[1], lo & 1))) break;
                    tc_fence_after();
                    drain(tbase + NT);
                    tc_fence_before();
                    mbar_arrive(&gempty[1]);
                    ++lo;
                }
            }
            if (!ok) break;
            const int mt = tile / a.ntiles, nt = tile - mt * a.ntiles;
            const int64_t col0 = (int64_t)nt * NT + quarter * hc;
            if (a.split) {
                float* dst = a.C + sg::part_slot(a, tile) * (128 * NT) + (int64_t)(quarter * hc) * 128 + r;
#pragma unroll
                for (int j = 0; j < kMaxCols; ++j)
                    if (j < hc) dst[j * 128] = sum[j];
            } else if (a.tma) {
                const int64_t rb = (int64_t)mt * 128 + g * 32;
#pragma unroll
                for (int j0 = 0; j0 < kMaxCols; j0 += 32) {
                    if (j0 < hc) {
                        if (lane == 0) bulk_wait_read<0>();      // the store before has read the buffer
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            *reinterpret_cast<float4*>(stage + lane * 32 + ((j >> 2) ^ (lane & 7)) * 4) =
                                make_float4(sum[j0 + j], sum[j0 + j + 1], sum[j0 + j + 2], sum[j0 + j + 3]);
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (lane == 0 && rb < a.M && col0 + j0 < a.N) {
                            tma_store_2d(&tm_c, (int32_t)(col0 + j0), (int32_t)rb, stage);
                            bulk_commit();
                        }
                    }
                }
            } else {
                const int64_t rb = (int64_t)mt * 128 + g * 32;
#pragma unroll
                for (int j0 = 0; j0 < kMaxCols; j0 += 32) {
                    if (j0 < hc) {
                        __syncwarp();
#pragma unroll
                        for (int j = 0; j < 32; ++j) stage[lane * kStagePitch + j] = sum[j0 + j];
                        __syncwarp();
                        const bool mine = j0 + lane < hc && col0 + j0 + lane < a.N;
                        float* dst = a.C + rb * a.ldc + col0 + j0 + lane;
#pragma unroll 8
                        for (int i = 0; i < 32; ++i)
                            if (mine && rb + i < a.M) dst[i * a.ldc] = stage[i * kStagePitch + lane];
                    }
                }
            }
        }
        if (a.tma && lane == 0) bulk_wait<0>();
    } else if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            sg::Pieces<GemmArgs> pc(a);
            int tile, c0, c1;
            int it = 0, slot = 0;
            uint32_t phase = 1;
            bool ok = true;
            while (ok && pc.next(a, &tile, &c0, &c1)) {
                const int mt = tile / a.ntiles, nt = tile - mt * a.ntiles;
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
        // per block.  hi hi comes last in a chunk's first block and first in its
        // last, so that ten MMAs lie between its accumulator's last use in one
        // chunk and its first in the next, time for the drain.
        sg::Pieces<GemmArgs> pc(a);
        int tile, c0, c1;
        int slot = 0, ch = 0, lo = 0;
        uint32_t phase = 0;
        bool ok = true;
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort, err, 2u)) != 0;
        };
        const uint32_t idesc = idesc_f16_f32(128, (uint32_t)NT) | kIdescBF16;
        constexpr uint32_t kPart = 8 * kKB * 2 / 16;
        const uint64_t ad = smem_desc(smem_u32(ring), 128, kGroupBytes, 0);
        const uint64_t bd = smem_desc(smem_u32(ring) + a.a_bytes, 128, kGroupBytes, 0);
        const uint32_t ahi = (uint32_t)(ad >> 32), bhi = (uint32_t)(bd >> 32), alo0 = (uint32_t)ad, blo0 = (uint32_t)bd;
        const uint32_t low = tmem + (uint32_t)NT;
        while (ok && pc.next(a, &tile, &c0, &c1)) {
            for (int c = c0; c < c1 && ok; ++c, ++ch) {
                const int nb = min(kChunkBlocks, a.kblocks - kChunkBlocks * c);
                const bool fresh = (c - c0) % kLowPeriod == 0;      // the lower products start a new sum
                const bool last = c + 1 == c1 || (c - c0 + 1) % kLowPeriod == 0;
                if (fresh && !(ok = wait(&gempty[1], (lo & 1) ^ 1))) break;
                for (int b = 0; b < nb; ++b) {
                    if (!(ok = wait(&full[slot], phase))) break;
                    tc_fence_after();
                    const uint32_t off = (uint32_t)slot * stage_bytes / 16;
                    const uint32_t al = alo0 + off, bl = blo0 + off;
                    const uint32_t acc = fresh && b == 0 ? 0u : 1u;
                    if (b > 0) {
                        if (elect_one()) {
                            mma_f16_col<kFill>(tmem, al, ahi, bl, bhi, idesc, 1u);                       // hi hi
                            if (b == nb - 1) mma_commit(&gfull[0]);
                            mma_f16_col<kUse>(low, al, ahi, bl + kPart, bhi, idesc, acc);                // hi mid
                            mma_f16_col<kLast>(low, al, ahi, bl + 2 * kPart, bhi, idesc, 1u);            // hi lo
                            mma_f16_col<kFill>(low, al + kPart, ahi, bl, bhi, idesc, 1u);                // mid hi
                            mma_f16_col<kLast>(low, al + kPart, ahi, bl + kPart, bhi, idesc, 1u);        // mid mid
                            mma_f16_col<kNoReuse>(low, al + 2 * kPart, ahi, bl, bhi, idesc, 1u);         // lo hi
                            mma_commit(&empty[slot]);
                        }
                        __syncwarp();
                    } else {
                        if (elect_one()) {
                            mma_f16_col<kNoReuse>(low, al + 2 * kPart, ahi, bl, bhi, idesc, acc);
                            mma_f16_col<kFill>(low, al + kPart, ahi, bl, bhi, idesc, 1u);
                            mma_f16_col<kLast>(low, al + kPart, ahi, bl + kPart, bhi, idesc, 1u);
                            mma_f16_col<kFill>(low, al, ahi, bl + kPart, bhi, idesc, 1u);
                            mma_f16_col<kLast>(low, al, ahi, bl + 2 * kPart, bhi, idesc, 1u);
                        }
                        __syncwarp();
                        if (!(ok = wait(&gempty[0], (ch & 1) ^ 1))) break;
                        tc_fence_after();
                        if (elect_one()) {
                            mma_f16_col<kNoReuse>(tmem, al, ahi, bl, bhi, idesc, 0u);
                            if (nb == 1) mma_commit(&gfull[0]);
                            mma_commit(&empty[slot]);
                        }
                        __syncwarp();
                    }
                    if (++slot == a.stages) {
                        slot = 0;
                        phase ^= 1;
                    }
                }
                if (!ok) break;
                if (last) {
                    if (elect_one()) mma_commit(&gfull[1]);
                    __syncwarp();
                    ++lo;
                }
            }
        }
        if (elect_one()) mma_commit(mma_done);
        __syncwarp();
        volatile int no_abort = 0;
        mbar_wait(mma_done, 0, &no_abort, err, 2u, 100000000ull);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, a.tmem_cols);
}

// The partial tiles of a split reduction, added in the order of the groups.
__global__ void __launch_bounds__(256) part_sum32_kernel(const float* __restrict__ part, int NT, int64_t ntiles,
                                                         int64_t chunks, int64_t Q, int64_t G, int group,
                                                         float* __restrict__ C, int64_t ldc, int64_t M, int64_t N,
                                                         const float* __restrict__ cscale) {
    __shared__ float sm[8][33];
    pdl_wait();
    pdl_trigger();
    const int64_t tile = blockIdx.x;
    const int64_t mt = tile / ntiles, nt = tile - mt * ntiles, u = tile / group * chunks;
    const int64_t p0 = sg::group_of_chunk(u, Q, G), p1 = sg::group_of_chunk(u + chunks - 1, Q, G);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    // 32 rows x 8 columns at a time, turned so that a row's columns are neighbours
    const int blocks = 4 * (NT / 8);
    for (int q = blockIdx.y; q < blocks; q += gridDim.y) {
        const int rb = (q & 3) * 32, cb = (q >> 2) * 8;
        const float* src = part + tile * (128 * NT) + (cb + ty) * 128 + rb + tx;
        const float s = sg::sum_parts<8>(0.0f, src, (int64_t)group * (128 * NT), p0, p1 + 1);
        __syncthreads();
        sm[ty][tx] = s;
        __syncthreads();
        const int64_t col = nt * NT + cb + (threadIdx.x & 7), row = mt * 128 + rb + (threadIdx.x >> 3);
        if (col < N && row < M)
            C[row * ldc + col] = __fmul_rn(sm[threadIdx.x & 7][threadIdx.x >> 3], cscale ? __ldg(cscale + col) : 1.0f);
    }
}

// ---------------------------------------------------------------- repair
struct RepairSide {
    const float* p;
    int64_t rs, cs, rows;
    const int* hard;
};

// Rows listed as hard: their part of C by binary32 FMAs, sums of at most 1024
// terms added up.  The tile follows from how many there are, so that a small
// result with a long reduction keeps the GPU at work: R x R entries a thread in
// tiles of 16 R, and for few entries (R = 0) tiles of 8 x 8 whose reduction is
// split over four threads.
template <int R>
__device__ __forceinline__ void repair32_body(const RepairSide& A, const RepairSide& B, int64_t K, float* C, int64_t ldc,
                                              const float* cscale, int64_t na, int64_t nb, float* As, float* Bs) {
    constexpr int T = R == 0 ? 8 : 16 * R, KS = 1024 / T, P = T + 1, E = R == 0 ? 1 : R, W = R == 0 ? 8 : 16;
    constexpr int XS = 256 / KS;
    const int64_t M = A.rows, N = B.rows;
    const int64_t ta = (na + T - 1) / T * ((N + T - 1) / T), tb = (nb + T - 1) / T * ((M + T - 1) / T);
    const int tid = threadIdx.x;
    const int part = R == 0 ? tid / 64 : 0;                        // quarter of a slab
    const int tx = tid % W, ty = R == 0 ? tid / 8 % 8 : tid / 16;
    for (int64_t t = blockIdx.x; t < ta + tb; t += gridDim.x) {
        const bool ga = t < ta;
        const int64_t u = ga ? t : t - ta;
        const int64_t other = ((ga ? N : M) + T - 1) / T;
        const int64_t l0 = u / other * T, o0 = (u % other) * T;
        const int64_t i0 = ga ? l0 : o0, j0 = ga ? o0 : l0;
        const int64_t ni = ga ? na : M, nj = ga ? N : nb;
        auto row_of = [&](int i) { return i0 + i >= ni ? -1 : ga ? __ldg(A.hard + 1 + i0 + i) : (int)(i0 + i); };
        auto col_of = [&](int j) { return j0 + j >= nj ? -1 : ga ? (int)(j0 + j) : __ldg(B.hard + 1 + j0 + j); };
        const int kk = tid % KS, x0 = tid / KS;                    // a thread stages four entries of each operand
        int ri[4], cj[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            ri[q] = row_of(x0 + q * XS);
            cj[q] = col_of(x0 + q * XS);
        }
        float acc[E][E], tot[E][E];
#pragma unroll
        for (int i = 0; i < E; ++i)
#pragma unroll
            for (int j = 0; j < E; ++j) acc[i][j] = tot[i][j] = 0.0f;
        float va[4], vb[4];
        auto load = [&](int64_t k0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                va[q] = ri[q] >= 0 && k0 + kk < K ? __ldg(A.p + ri[q] * A.rs + (k0 + kk) * A.cs) : 0.0f;
                vb[q] = cj[q] >= 0 && k0 + kk < K ? __ldg(B.p + cj[q] * B.rs + (k0 + kk) * B.cs) : 0.0f;
            }
        };
        load(0);
        for (int64_t k0 = 0; k0 < K; k0 += KS) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                As[kk * P + x0 + q * XS] = va[q];
                Bs[kk * P + x0 + q * XS] = vb[q];
            }
            __syncthreads();
            if (k0 + KS < K) load(k0 + KS);                        // in flight over this slab's FMAs
            const int kn = (int)min((int64_t)KS, K - k0);
            const int kb = R == 0 ? part * (KS / 4) : 0, ke = R == 0 ? min(kn, kb + KS / 4) : kn;
#pragma unroll 4
            for (int k = kb; k < ke; ++k) {
                float x[E], y[E];
#pragma unroll
                for (int i = 0; i < E; ++i) x[i] = As[k * P + ty + W * i];
#pragma unroll
                for (int j = 0; j < E; ++j) y[j] = Bs[k * P + tx + W * j];
#pragma unroll
                for (int i = 0; i < E; ++i)
#pragma unroll
                    for (int j = 0; j < E; ++j) acc[i][j] = fmaf(x[i], y[j], acc[i][j]);
            }
            __syncthreads();
            if (((k0 + KS) & 1023) == 0 || k0 + KS >= K) {
#pragma unroll
                for (int i = 0; i < E; ++i)
#pragma unroll
                    for (int j = 0; j < E; ++j) {
                        tot[i][j] += acc[i][j];
                        acc[i][j] = 0.0f;
                    }
            }
        }
        if (R == 0) {
            As[tid] = tot[0][0];
            __syncthreads();
            tot[0][0] = ((As[tid & 63] + As[64 + (tid & 63)]) + As[128 + (tid & 63)]) + As[192 + (tid & 63)];
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
                if (col >= 0) C[row * ldc + col] = cscale ? tot[i][j] * __ldg(cscale + col) : tot[i][j];
            }
        }
    }
}

__global__ void __launch_bounds__(256, 2) repair32_kernel(const __grid_constant__ RepairSide A,
                                                          const __grid_constant__ RepairSide B, int64_t K,
                                                          float* __restrict__ C, int64_t ldc,
                                                          const float* __restrict__ cscale) {
    __shared__ float As[128 * 9], Bs[128 * 9];                     // the largest of all R, with padding
    pdl_wait();
    pdl_trigger();
    const int64_t M = A.rows, N = B.rows, na = A.hard[0], nb = na == M ? 0 : B.hard[0];   // every row of A: all of C
    if (na + nb == 0) return;
    auto tiles = [&](int T) { return (na + T - 1) / T * ((N + T - 1) / T) + (nb + T - 1) / T * ((M + T - 1) / T); };
    const int64_t grid = gridDim.x;
    if (tiles(64) >= grid) repair32_body<4>(A, B, K, C, ldc, cscale, na, nb, As, Bs);
    else if (tiles(32) >= grid) repair32_body<2>(A, B, K, C, ldc, cscale, na, nb, As, Bs);
    else if (tiles(16) >= 4 * grid) repair32_body<1>(A, B, K, C, ldc, cscale, na, nb, As, Bs);
    else repair32_body<0>(A, B, K, C, ldc, cscale, na, nb, As, Bs);
}

int64_t n_tiles(int64_t rows, bool splitk) { return (rows + n_tile(rows, splitk) - 1) / n_tile(rows, splitk); }

}  // namespace

lrc_status split(const Operand* const* ops, int count, cudaStream_t s) {
    Jobs js{};
    int64_t bl = 0;
    for (int i = 0; i < count; ++i) {
        const Operand& o = *ops[i];
        Job& j = js.j[js.n++];
        j.p = o.p;
        j.rs = o.rs;
        j.cs = o.cs;
        j.rows = o.rows;
        j.K = o.K;
        j.img_rows = image_rows(o.rows);
        j.kblocks = image_blocks(o.K);
        j.vec = o.cs == 1 && o.rs % 4 == 0 && aligned16(o.p);
        j.limit = o.second ? kSecondLimit : kFirstLimit;
        j.img = o.img;
        j.hard = o.hard;
        j.kparts = (int)((j.kblocks * kKB + kJobCols - 1) / kJobCols);
        j.b0 = bl;
        bl += (j.img_rows + 31) / 32 * j.kparts;
    }
    if (bl > 0x7fffffff) {
        set_error("split product: operand too large");
        return LRC_ERR_UNSUPPORTED;
    }
    const cudaError_t e = launch_pdl(parts_kernel, dim3((unsigned)bl), dim3(256), 0, s, js);
    if (e != cudaSuccess) return cuda_fail(e, "parts_kernel launch");
    return after_launch("parts_kernel");
}

size_t part_bytes(int64_t M, int64_t N) {
    return (((M + 127) / 128 * n_tiles(N, true) + sm_count()) * 128 * (size_t)n_tile(N, true) * 4 + 255) & ~(size_t)255;
}

lrc_status product(const Operand& A, const Operand& B, float* C, int64_t ldc, const float* cscale, bool splitk,
                   float* part, cudaStream_t s) {
    const int NT = n_tile(B.rows, splitk);
    const int64_t tiles = (A.rows + 127) / 128 * n_tiles(B.rows, splitk);
    if (tiles > 0x3fffffff || A.K > (1ll << 30)) {
        set_error("split product too large (%lld tiles)", (long long)tiles);
        return LRC_ERR_UNSUPPORTED;
    }
    GemmArgs a{};
    a.A = A.img;
    a.B = B.img;
    a.C = splitk ? part : C;
    a.ldc = ldc;
    a.M = A.rows;
    a.N = B.rows;
    a.ntiles = (int)n_tiles(B.rows, splitk);
    a.tiles = (int)tiles;
    a.kblocks = (int)image_blocks(A.K);
    a.chunks = (a.kblocks + kChunkBlocks - 1) / kChunkBlocks;
    a.split = splitk;
    a.NT = NT;
    a.a_block = image_rows(A.rows) / 8 * kGroupBytes;
    a.b_block = image_rows(B.rows) / 8 * kGroupBytes;
    a.a_bytes = 128 / 8 * kGroupBytes;
    a.b_bytes = (uint32_t)(NT / 8 * kGroupBytes);
    CUtensorMap tm{};
    a.tma = !splitk && ldc % 4 == 0 && aligned16(C);
    lrc_status st;
    if (a.tma && (st = encode_map_2d(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, C, B.rows, A.rows, ldc * 4, 32, 32, true,
                                     "product32 output")) != LRC_OK)
        return st;
    const size_t staging = splitk ? 0 : (size_t)kEpiWarps * kStageBytes;
    a.stages = (int)std::min<int64_t>(8, (int64_t)(227 * 1024 - kCtrlBytes - staging) / (a.a_bytes + a.b_bytes));
    uint32_t cols = 64;
    // (a drain reads 16 columns at a time, past the last quarter's end)
    while (cols < (uint32_t)(2 * NT + (NT % 64 ? 16 : 0))) cols *= 2;
    a.tmem_cols = cols;
    const int64_t sms = sm_count();
    a.group = splitk && (int64_t)a.ntiles * 8 <= sms ? a.ntiles : 1;
    const int64_t Q = tiles / a.group * a.chunks;
    const int64_t groups = std::min<int64_t>(Q, sms / a.group);
    const int64_t grid = splitk ? groups * a.group : std::min<int64_t>(tiles, sms);
    const size_t smem = kCtrlBytes + (size_t)a.stages * (a.a_bytes + a.b_bytes) + staging;
    cudaError_t e = cudaFuncSetAttribute(product32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return cuda_fail(e, "product32_kernel smem attribute");
    e = launch_pdl(product32_kernel, dim3((unsigned)grid), dim3(kThreads), smem, s, a, tm);
    if (e != cudaSuccess) return cuda_fail(e, "product32_kernel launch");
    st = after_launch("product32_kernel");
    if (st != LRC_OK) return st;
    if (splitk) {
        const unsigned gy = (unsigned)std::max<int64_t>(1, std::min<int64_t>(NT / 2, 8 * sms / tiles));
        e = launch_pdl(part_sum32_kernel, dim3((unsigned)tiles, gy), dim3(256), 0, s, (const float*)part, NT,
                       (int64_t)a.ntiles, (int64_t)a.chunks, Q, groups, a.group, C, ldc, A.rows, B.rows, cscale);
        if (e != cudaSuccess) return cuda_fail(e, "part_sum32_kernel launch");
        if ((st = after_launch("part_sum32_kernel")) != LRC_OK) return st;
    }
    e = launch_pdl(repair32_kernel, dim3((unsigned)(2 * sms)), dim3(256), 0, s,
                   RepairSide{A.p, A.rs, A.cs, A.rows, A.hard}, RepairSide{B.p, B.rs, B.cs, B.rows, B.hard}, A.K, C, ldc,
                   cscale);
    if (e != cudaSuccess) return cuda_fail(e, "repair32_kernel launch");
    return after_launch("repair32_kernel");
}

}  // namespace sg32

uint32_t take_split32_error() {
    unsigned int v = 0;
    if (cudaMemcpyFromSymbol(&v, sg32::g_err_split32, sizeof v) != cudaSuccess) return 0xffffffffu;
    if (v) {
        const unsigned int z = 0;
        cudaMemcpyToSymbol(sg32::g_err_split32, &z, sizeof z);
    }
    return v;
}

}  // namespace lrc
