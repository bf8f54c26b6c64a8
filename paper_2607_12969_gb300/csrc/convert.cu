// convert.cu -- factor rounding / packing (binary64 -> binary32 / binary16 /
// bfloat16) and exact widening back to binary64.
//
// Rounding is the hardware conversion cvt.rn.{f32,f16,bf16}.f64: IEEE 754
// round-to-nearest-even directly from binary64 (no intermediate format),
// subnormals kept (no .ftz), overflow to infinity; the 16-bit formats take it
// only where the result is no normal number, and integer operations with the
// same result elsewhere (round16).  The kernels are HBM-bound streams: each
// thread converts a group of 8 consecutive elements of one row with 128-bit
// loads and stores where the row pitch allows it; a matrix whose elements lie
// in one run is converted without row arithmetic (round_run_kernel).
#include <cuda_fp16.h>

#include "common.cuh"

namespace lrc {
namespace {

constexpr int kThreads = 256;
constexpr int kGroup = 8;

__device__ __forceinline__ uint16_t cvt_f16(double x) {
    uint16_t h;
    asm("cvt.rn.f16.f64 %0, %1;" : "=h"(h) : "d"(x));
    return h;
}
__device__ __forceinline__ uint16_t cvt_bf16(double x) {
    uint16_t h;
    asm("cvt.rn.bf16.f64 %0, %1;" : "=h"(h) : "d"(x));
    return h;
}
__device__ __forceinline__ float cvt_f32(double x) {
    float f;
    asm("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(x));
    return f;
}
__device__ __forceinline__ double widen_f16(uint16_t h) {
    double d;
    asm("cvt.f64.f16 %0, %1;" : "=d"(d) : "h"(h));
    return d;
}

// Rounding to a 16-bit format by integer operations, for zeros and for results
// in the normal exponents (or that overflow by rounding up): the dropped bits of
// the significand's upper word, with one bit for whether the lower word is zero,
// rounded to nearest even into the encoding, whose carry reaches the exponent as
// it should.  MANT: stored significand bits, BIAS: exponent bias; `special` is
// set for every other input.
template <int MANT, int BIAS>
__device__ __forceinline__ uint32_t round16(double x, bool* special) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    constexpr int drop = 20 - MANT;
    const uint32_t a = hi & 0x7fffffffu;
    const uint32_t s = a | (lo != 0 ? 1u : 0u);
    const uint32_t h = ((s + (1u << (drop - 1)) - 1u + ((s >> drop) & 1u)) >> drop) - ((uint32_t)(1023 - BIAS) << MANT);
    *special |= s != 0 && (a >> 20) - (uint32_t)(1024 - BIAS) >= (uint32_t)(2 * BIAS);
    return (s != 0 ? h : 0u) | ((hi >> 16) & 0x8000u);
}

// A group in a 16-bit format (FMT 2 or 3).  The conversion instructions from
// binary64 issue about two a clock on an SM: 4096 x 16384 elements took 117 us
// with them however they were loaded, and take 96 us (7.0 TB/s) without.  The
// vote makes the branch a real one: with `special` alone the conversions are
// issued for every group, switched off by a predicate, and the kernel takes
// 130 us.  With a special value in every warp it takes the 117 us.
template <int FMT>
__device__ __forceinline__ void round_group(const double* v, uint32_t* h) {
    bool special = false;
#pragma unroll
    for (int j = 0; j < kGroup; ++j)
        h[j] = FMT == 2 ? round16<10, 15>(v[j], &special) : round16<7, 127>(v[j], &special);
    if (__any_sync(__activemask(), special)) {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) h[j] = FMT == 2 ? cvt_f16(v[j]) : cvt_bf16(v[j]);
    }
}
__device__ __forceinline__ uint4 pack_group(const uint32_t* h) {
    return make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
}

// Four doubles in one 32-byte load (p on a 32-byte boundary), read once.
__device__ __forceinline__ void load4(const double* p, double* v) {
    asm volatile("ld.global.L1::no_allocate.v4.f64 {%0,%1,%2,%3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
}

// A source whose elements lie in one run of whole groups, to a 16-bit format:
// one group a thread and as many blocks as that takes.  Two or four groups in
// flight in a thread gave nothing (96.0 us either way), a grid of resident
// blocks that strides over the groups cost 4 us.
template <int FMT>
__global__ void __launch_bounds__(kThreads)
round_run_kernel(const double* __restrict__ src, uint16_t* __restrict__ dst, int64_t groups) {
    const int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (g >= groups) return;
    double v[kGroup];
    load4(src + g * kGroup, v);
    load4(src + g * kGroup + 4, v + 4);
    uint32_t h[kGroup];
    round_group<FMT>(v, h);
    __stcs(reinterpret_cast<uint4*>(dst) + g, pack_group(h));
}

// FMT: 0 = binary64 copy, 1 = binary32, 2 = binary16, 3 = bfloat16
template <int FMT>
__global__ void __launch_bounds__(kThreads)
round_pack_kernel(const double* __restrict__ src, int64_t cols, int64_t ld_src,
                  void* __restrict__ dst, int64_t ld_dst, int64_t groups_per_row,
                  int64_t total_groups, bool vec_src, bool vec_dst) {
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x; g < total_groups; g += stride) {
        const int64_t r = g / groups_per_row;
        const int64_t c0 = (g - r * groups_per_row) * kGroup;
        const double* srow = src + r * ld_src;
        double v[kGroup];
        if (vec_src && c0 + kGroup <= cols) {
#pragma unroll
            for (int j = 0; j < kGroup; j += 2) {
                const double2 p = __ldcs(reinterpret_cast<const double2*>(srow + c0 + j));
                v[j] = p.x;
                v[j + 1] = p.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < kGroup; ++j) v[j] = (c0 + j < cols) ? __ldcs(srow + c0 + j) : 0.0;
        }
        const bool full = vec_dst && (c0 + kGroup <= ld_dst);
        if (FMT == 2 || FMT == 3) {
            uint16_t* drow = static_cast<uint16_t*>(dst) + r * ld_dst;
            uint32_t h[kGroup];
            round_group<FMT == 3 ? 3 : 2>(v, h);
            if (full) {
                __stcs(reinterpret_cast<uint4*>(drow + c0), pack_group(h));
            } else {
                for (int j = 0; j < kGroup; ++j)
                    if (c0 + j < ld_dst) drow[c0 + j] = (uint16_t)h[j];
            }
        } else if (FMT == 1) {
            float* drow = static_cast<float*>(dst) + r * ld_dst;
            float f[kGroup];
#pragma unroll
            for (int j = 0; j < kGroup; ++j) f[j] = cvt_f32(v[j]);
            if (full) {
                __stcs(reinterpret_cast<float4*>(drow + c0), make_float4(f[0], f[1], f[2], f[3]));
                __stcs(reinterpret_cast<float4*>(drow + c0 + 4), make_float4(f[4], f[5], f[6], f[7]));
            } else {
                for (int j = 0; j < kGroup; ++j)
                    if (c0 + j < ld_dst) drow[c0 + j] = f[j];
            }
        } else {
            double* drow = static_cast<double*>(dst) + r * ld_dst;
            if (full) {
#pragma unroll
                for (int j = 0; j < kGroup; j += 2)
                    __stcs(reinterpret_cast<double2*>(drow + c0 + j), make_double2(v[j], v[j + 1]));
            } else {
                for (int j = 0; j < kGroup; ++j)
                    if (c0 + j < ld_dst) drow[c0 + j] = v[j];
            }
        }
    }
}

// Exact binary32 -> binary64 from the bit fields: normal numbers and zeros
// take integer operations only (the exponent rebias and significand shift of
// the IEEE 754 formats); subnormals, infinities and NaNs take the conversion
// instruction.
__device__ __forceinline__ double widen_f32(float f) {
    const uint32_t u = __float_as_uint(f);
    const uint32_t e = (u >> 23) & 0xffu;
    const unsigned long long sign = (unsigned long long)(u & 0x80000000u) << 32;
    if (e != 0u && e != 0xffu)
        return __longlong_as_double((long long)(sign | ((unsigned long long)(e + 896u) << 52) |
                                                ((unsigned long long)(u & 0x7fffffu) << 29)));
    if ((u & 0x7fffffffu) == 0u) return __longlong_as_double((long long)sign);
    return (double)f;
}

// FMT as above; dst is binary64.  Each thread widens a group of 8 elements of
// one row: one 16-byte (binary16) or two (binary32) loads, four 16-byte stores
// when the row pitches allow it.
template <int FMT>
__global__ void __launch_bounds__(kThreads)
widen_kernel(const void* __restrict__ src, int64_t cols, int64_t ld_src, double* __restrict__ dst,
             int64_t ld_dst, int64_t groups_per_row, int64_t total_groups, bool vec_src, bool vec_dst) {
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    for (int64_t g = (int64_t)blockIdx.x * kThreads + threadIdx.x; g < total_groups; g += stride) {
        const int64_t r = g / groups_per_row;
        const int64_t c0 = (g - r * groups_per_row) * kGroup;
        double v[kGroup];
        if (vec_src && c0 + kGroup <= cols) {
            if (FMT == 2 || FMT == 3) {
                const uint4 q = __ldcs(reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(src) + r * ld_src + c0));
                const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    // a bfloat16 value is the binary32 number with the same upper 16 bits
                    const float2 f = FMT == 2 ? __half22float2(*reinterpret_cast<const __half2*>(&w[j]))
                                              : make_float2(__uint_as_float(w[j] << 16), __uint_as_float(w[j] & 0xffff0000u));
                    v[2 * j] = widen_f32(f.x);
                    v[2 * j + 1] = widen_f32(f.y);
                }
            } else if (FMT == 1) {
                const float4* p = reinterpret_cast<const float4*>(static_cast<const float*>(src) + r * ld_src + c0);
                const float4 a = __ldcs(p), b = __ldcs(p + 1);
                v[0] = widen_f32(a.x); v[1] = widen_f32(a.y); v[2] = widen_f32(a.z); v[3] = widen_f32(a.w);
                v[4] = widen_f32(b.x); v[5] = widen_f32(b.y); v[6] = widen_f32(b.z); v[7] = widen_f32(b.w);
            } else {
                const double2* p = reinterpret_cast<const double2*>(static_cast<const double*>(src) + r * ld_src + c0);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const double2 t = __ldcs(p + j);
                    v[2 * j] = t.x;
                    v[2 * j + 1] = t.y;
                }
            }
        } else {
#pragma unroll
            for (int j = 0; j < kGroup; ++j) {
                const int64_t c = c0 + j;
                double x = 0.0;
                if (c < cols) {
                    if (FMT == 2) x = widen_f16(static_cast<const uint16_t*>(src)[r * ld_src + c]);
                    else if (FMT == 3)
                        x = widen_f32(__uint_as_float((uint32_t)static_cast<const uint16_t*>(src)[r * ld_src + c] << 16));
                    else if (FMT == 1) x = (double)static_cast<const float*>(src)[r * ld_src + c];
                    else x = static_cast<const double*>(src)[r * ld_src + c];
                }
                v[j] = x;
            }
        }
        double* drow = dst + r * ld_dst;
        if (vec_dst && c0 + kGroup <= ld_dst) {
#pragma unroll
            for (int j = 0; j < kGroup; j += 2)
                __stcs(reinterpret_cast<double2*>(drow + c0 + j), make_double2(v[j], v[j + 1]));
        } else {
            for (int j = 0; j < kGroup; ++j)
                if (c0 + j < ld_dst) drow[c0 + j] = v[j];
        }
    }
}

int grid_for(int64_t groups) {
    const int64_t want = (groups + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)sm_count() * 8;
    return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}

}  // namespace

lrc_status launch_round(const double* src, int64_t rows, int64_t cols, int64_t ld_src, void* dst,
                        int64_t ld_dst, lrc_fmt fmt, cudaStream_t s) {
    const int64_t gpr = (ld_dst + kGroup - 1) / kGroup;
    const int64_t total = rows * gpr;
    const bool vec_src = (ld_src % 2) == 0;
    const int grid = grid_for(total);
    const int64_t run_blocks = (total + kThreads - 1) / kThreads;
    if (storage_bytes(fmt) == 2 && cols == ld_src && cols == ld_dst && cols % kGroup == 0 && total > 0 &&
        run_blocks <= 0x7fffffff && reinterpret_cast<uintptr_t>(src) % 32 == 0 &&
        reinterpret_cast<uintptr_t>(dst) % 16 == 0) {
        uint16_t* out = static_cast<uint16_t*>(dst);
        if (fmt == LRC_BF16) round_run_kernel<3><<<(unsigned)run_blocks, kThreads, 0, s>>>(src, out, total);
        else round_run_kernel<2><<<(unsigned)run_blocks, kThreads, 0, s>>>(src, out, total);
        return after_launch("round_run_kernel");
    }
    switch (fmt) {
        case LRC_F64:
            round_pack_kernel<0><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total,
                                                            vec_src, (ld_dst % 2) == 0);
            break;
        case LRC_F32:
            round_pack_kernel<1><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total,
                                                            vec_src, (ld_dst % 4) == 0);
            break;
        case LRC_BF16:
            round_pack_kernel<3><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total,
                                                            vec_src, (ld_dst % 8) == 0);
            break;
        default:
            round_pack_kernel<2><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total,
                                                            vec_src, (ld_dst % 8) == 0);
            break;
    }
    return after_launch("round_pack_kernel");
}

lrc_status launch_widen(const void* src, lrc_fmt fmt, int64_t rows, int64_t cols, int64_t ld_src,
                        double* dst, int64_t ld_dst, cudaStream_t s) {
    const int64_t gpr = (ld_dst + kGroup - 1) / kGroup;
    const int64_t total = rows * gpr;
    const int grid = grid_for(total);
    const int64_t e = storage_bytes(fmt);
    // 16-byte vectors: row starts (base and pitch) on 16-byte boundaries
    const bool vec_src = (reinterpret_cast<uintptr_t>(src) % 16 == 0) && ((ld_src * e) % 16 == 0);
    const bool vec_dst = (reinterpret_cast<uintptr_t>(dst) % 16 == 0) && (ld_dst % 2 == 0);
    switch (fmt) {
        case LRC_F64:
            widen_kernel<0><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total, vec_src, vec_dst);
            break;
        case LRC_F32:
            widen_kernel<1><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total, vec_src, vec_dst);
            break;
        case LRC_BF16:
            widen_kernel<3><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total, vec_src, vec_dst);
            break;
        default:
            widen_kernel<2><<<grid, kThreads, 0, s>>>(src, cols, ld_src, dst, ld_dst, gpr, total, vec_src, vec_dst);
            break;
    }
    return after_launch("widen_kernel");
}

}  // namespace lrc
