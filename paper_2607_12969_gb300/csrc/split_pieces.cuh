// split_pieces.cuh -- how the persistent product kernels of split_gemm.cu and
// split_gemm32.cu walk their tiles.
#pragma once

#include <stdint.h>

namespace lrc {
namespace sg {

// The (tile, chunk range) pieces of a CTA, in order.  A split reduction is cut
// over groups of `group` CTAs, one per tile of B: a group walks one range of
// (tile of A, chunk), laid end to end, so that its CTAs read the same blocks of
// A at about the same time and only the first read comes from HBM.
template <typename Args>
struct Pieces {
    int left, t, c, step;      // split: chunks left, first chunk of the next piece
    __device__ explicit Pieces(const Args& a) {
        if (a.split) {
            const int groups = gridDim.x / a.group, gi = blockIdx.x / a.group;
            const int64_t Q = (int64_t)(a.tiles / a.group) * a.chunks;
            const int64_t q0 = Q * gi / groups, q1 = Q * (gi + 1) / groups;
            const int mt = (int)(q0 / a.chunks);
            t = mt * a.group + (int)(blockIdx.x - gi * a.group);
            c = (int)(q0 - (int64_t)mt * a.chunks);
            left = (int)(q1 - q0);
            step = a.group;
        } else {
            t = blockIdx.x;
            c = 0;
            step = gridDim.x;
            left = t < a.tiles ? 1 : 0;
        }
    }
    // false: no piece left
    __device__ bool next(const Args& a, int* tile, int* c0, int* c1) {
        if (left <= 0) return false;
        *tile = t;
        *c0 = c;
        *c1 = a.chunks;
        t += step;
        if (a.split) {
            *c1 = min(a.chunks, c + left);
            left -= *c1 - c;
            c = 0;
        } else {
            left = t < a.tiles ? 1 : 0;
        }
        return true;
    }
};
// Partial tile of a piece: distinct for every (group, tile).
template <typename Args>
__device__ __forceinline__ int64_t part_slot(const Args& a, int tile) {
    return (int64_t)(blockIdx.x / a.group) * a.group + tile;
}

// The group that chunk u (of all tiles of A) falls to.
__host__ __device__ __forceinline__ int64_t group_of_chunk(int64_t u, int64_t Q, int64_t G) {
    return ((u + 1) * G + Q - 1) / Q - 1;
}

// p0 .. p1 - 1 of the partial tiles added to s in order, kAhead loads in flight
// also for the last ones (an unrolled loop takes what is left over one at a
// time: the 38 partial tiles of an entry were ten loads waited for in turn).
// Past the end the last load is repeated and zero added; a condition on the load
// or the sum makes the compiler wait for each load in turn.
template <int kAhead, typename T>
__device__ __forceinline__ T sum_parts(T s, const T* __restrict__ part, int64_t step, int64_t p0, int64_t p1) {
    int left = (int)(p1 - p0);
    for (const T* at = part + p0 * step; left > 0; left -= kAhead, at += kAhead * step) {
        T v[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) v[i] = __ldg(at + min(i, left - 1) * step);   // no branch between the loads
#pragma unroll
        for (int i = 0; i < kAhead; ++i) s += i < left ? v[i] : T(0);
    }
    return s;
}

}  // namespace sg
}  // namespace lrc
