// tt_chain.cu -- TT reconstruction as a chain of matrix products (Sec. 5.1:
// T(i_1..i_d) = G_1(i_1)...G_d(i_d); Sec. 7.5, Eq. gpu_tt_reconstruction:
// B_l = Z_{l-1} K_l) contracted from both ends toward one bond c:
//   left   Z(1) = G_1,      Z(j+1) = Z(j) K_j            (P_j x r_j rows)
//   right  S(d) = G_d,      S(j)   = K'_j S(j+1)         (r_{j-1} x Q_j)
//   output T = Z(c) S(c+1), a (n_1...n_c) x (n_{c+1}...n_d) matrix, which is
//          the C-order tensor.
// K_j is core j viewed as r_{j-1} x (n_j r_j) and K'_j the same core viewed
// as (r_{j-1} n_j) x r_j -- both are the stored C-order array, so every
// reshape is free.  The bond c minimises the multiply count; the last
// product writes the output and carries nearly all the work.  For the 16^6
// tensor with ranks (1,16,26,26,26,16,1) the chain meets at the middle bond:
// 0.88 GFLOP, against 1.50 GFLOP for the left-to-right chain.
//
// Every product runs on the product kernels of gemm_cc.cu (register-tiled
// binary32, DFMA-bound binary64); intermediates live in the stream's
// workspace (two buffers per side, alternating).
#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "split_gemm.cuh"
#include "split_gemm32.cuh"

namespace lrc {

namespace {

struct ChainPlan {
    int c;                  // bond: left cores 0..c-1, right cores c..d-1 (0-based)
    double flops;
};

// Multiply-adds x 2 of the chain that meets at bond c.
double chain_flops(const TTShape& sh, int c) {
    const int d = sh.d;
    double f = 0.0, P = (double)sh.dims[0];
    for (int j = 1; j <= c - 1; ++j) {
        f += 2.0 * P * (double)sh.ranks[j] * (double)sh.dims[j] * (double)sh.ranks[j + 1];
        P *= (double)sh.dims[j];
    }
    double Q = (double)sh.dims[d - 1];
    for (int j = d - 2; j >= c; --j) {
        f += 2.0 * (double)sh.ranks[j] * (double)sh.dims[j] * (double)sh.ranks[j + 1] * Q;
        Q *= (double)sh.dims[j];
    }
    return f + 2.0 * P * Q * (double)sh.ranks[c];
}

ChainPlan plan_chain(const TTShape& sh) {
    ChainPlan best{sh.d - 1, INFINITY};
    for (int c = 1; c <= sh.d - 1; ++c) {
        const double f = chain_flops(sh, c);
        if (f <= best.flops) best = ChainPlan{c, f};   // ties: the larger c (fewer right products)
    }
    return best;
}

size_t round256(size_t bytes) { return (bytes + 255) / 256 * 256; }

}  // namespace

double tt_chain_flops(const TTShape& sh) { return plan_chain(sh).flops; }

int tt_chain_bond(const TTShape& sh) { return plan_chain(sh).c; }

namespace {

lrc_status product(const float* A, int64_t lda, const float* B, int64_t ldb, float* C, int64_t ldc, int64_t M,
                   int64_t N, int64_t K, cudaStream_t s) {
    return gemm_cc_f32(A, lda, B, ldb, false, C, ldc, M, N, K, 1, 0, s);
}
lrc_status product(const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc, int64_t M,
                   int64_t N, int64_t K, cudaStream_t s) {
    return gemm_cc_f64(A, lda, B, ldb, C, ldc, M, N, K, s);
}

// Output products of binary32 chains go through bfloat16 parts from here on.
// Measured, parts / FMA kernel: 512 x 512 x 224, ranks 70, 52 (6.1e9) 147 / 249 us,
// 700 x 500 x 300, ranks 80, 40 (8.4e9) 207 / 368, 2048^2, rank 300 (2.5e9) 27 / 70.
// Below it the parts gain too (4096^2, rank 68 (2.3e9) 33 / 61, 10^5 x 64, rank 100
// (1.3e9) 49 / 72, 256^3, ranks 70 (2.3e9) 64 / 86), so it could lie lower.
constexpr double kPartsFlops = 2.5e9;

// tc_final (binary32 only): a smaller output product on the tensor cores through
// the scaled binary16 split (LRC_F32_TC) when the product kernel takes it.
template <typename T>
lrc_status launch_chain(const TTShape& sh, T* out, cudaStream_t s, bool tc_final = false) {
    const int d = sh.d;
    const int c = plan_chain(sh).c;
    const T* const* G = reinterpret_cast<const T* const*>(sh.cores);
    // P[j]: rows of Z(j); Q[j]: columns of S(j) (0-based core index j)
    int64_t P[17] = {0}, Q[17] = {0};
    P[1] = sh.dims[0];
    for (int j = 1; j <= c - 1; ++j) P[j + 1] = P[j] * sh.dims[j];
    Q[d - 1] = sh.dims[d - 1];
    for (int j = d - 2; j >= c; --j) Q[j] = sh.dims[j] * Q[j + 1];
    size_t lsz[2] = {0, 0}, rsz[2] = {0, 0};
    for (int j = 2; j <= c; ++j) {
        const size_t b = round256((size_t)P[j] * (size_t)sh.ranks[j] * sizeof(T));
        if (b > lsz[j & 1]) lsz[j & 1] = b;
    }
    for (int j = c; j <= d - 2; ++j) {
        const size_t b = round256((size_t)sh.ranks[j] * (size_t)Q[j] * sizeof(T));
        if (b > rsz[j & 1]) rsz[j & 1] = b;
    }
    unsigned char* ws = nullptr;
    const int64_t rc = sh.ranks[c];
    const size_t sides = lsz[0] + lsz[1] + rsz[0] + rsz[1];
    // binary32: a large output product in bfloat16 parts (split_gemm32.cu), where
    // there is workspace for them
    sg32::Operand oz{nullptr, rc, 1, P[c], rc, false, nullptr, nullptr};
    sg32::Operand os{nullptr, 1, Q[c], Q[c], rc, true, nullptr, nullptr};
    const size_t zi = round256(sg32::image_bytes(P[c], rc)), si = round256(sg32::image_bytes(Q[c], rc));
    bool parts = sizeof(T) == 4 && 2.0 * (double)P[c] * (double)Q[c] * (double)rc >= kPartsFlops &&
                 std::max(P[c], Q[c]) < ((int64_t)1 << 31);      // (rows are numbered in 32 bits)
    if (parts) {
        void* p = nullptr;
        const lrc_status st = stream_workspace_try(
            s, sides + zi + si + sg32::hard_bytes(P[c]) + sg32::hard_bytes(Q[c]), &p);
        if (st != LRC_OK) return st;
        parts = p != nullptr;
        ws = static_cast<unsigned char*>(p);
    }
    const bool tc = !parts && tc_final && sizeof(T) == 4 && split_product_fits(P[c], Q[c], rc);
    const size_t tsz = tc ? round256(split_product_bytes(P[c], Q[c], rc)) : 0;
    if (!parts && sides + tsz > 0) {
        void* p = nullptr;
        lrc_status st = stream_workspace(s, sides + tsz, &p);
        if (st != LRC_OK) return st;
        ws = static_cast<unsigned char*>(p);
    }
    T* L[2] = {reinterpret_cast<T*>(ws), reinterpret_cast<T*>(ws + lsz[0])};
    T* R[2] = {reinterpret_cast<T*>(ws + lsz[0] + lsz[1]), reinterpret_cast<T*>(ws + lsz[0] + lsz[1] + rsz[0])};
    lrc_status st = LRC_OK;
    const T* Z = G[0];   // Z(1) = G_1: n_1 x r_1
    for (int j = 1; j <= c - 1; ++j) {
        const int64_t w = sh.dims[j] * sh.ranks[j + 1];
        T* dst = L[(j + 1) & 1];
        if ((st = product(Z, sh.ranks[j], G[j], w, dst, w, P[j], w, sh.ranks[j], s)) != LRC_OK) return st;
        Z = dst;
    }
    const T* S = G[d - 1];   // S(d) = G_d: r_{d-1} x n_d
    for (int j = d - 2; j >= c; --j) {
        T* dst = R[j & 1];
        if ((st = product(G[j], sh.ranks[j + 1], S, Q[j + 1], dst, Q[j + 1], sh.ranks[j] * sh.dims[j], Q[j + 1],
                          sh.ranks[j + 1], s)) != LRC_OK)
            return st;
        S = dst;
    }
    if constexpr (sizeof(T) == 4) {
        if (parts) {
            unsigned char* q = ws + sides;
            oz.p = Z;
            os.p = S;
            oz.img = q;
            os.img = q + zi;
            oz.hard = reinterpret_cast<int*>(q + zi + si);
            os.hard = reinterpret_cast<int*>(q + zi + si + sg32::hard_bytes(P[c]));
            const cudaError_t e = cudaMemsetAsync(oz.hard, 0, sg32::hard_bytes(P[c]) + sg32::hard_bytes(Q[c]), s);
            if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync (row lists)");
            const sg32::Operand* ops[2] = {&oz, &os};
            if ((st = sg32::split(ops, 2, s)) != LRC_OK) return st;
            return sg32::product(oz, os, out, Q[c], nullptr, false, nullptr, s);
        }
        // Z is P x r (row pitch r), S is r x Q (row pitch Q): B = S^T
        if (tc)
            return launch_split_product(Z, rc, 1, S, 1, Q[c], P[c], Q[c], rc,
                                        ws + lsz[0] + lsz[1] + rsz[0] + rsz[1], out, s);
    }
    return product(Z, sh.ranks[c], S, Q[c], out, Q[c], P[c], Q[c], sh.ranks[c], s);
}

}  // namespace

lrc_status launch_tt_chain_f32(const TTShape& sh, float* out, cudaStream_t s) {
    bool handled = false;
    lrc_status st = launch_tt_split_f32(sh, out, s, &handled);
    if (st != LRC_OK || handled) return st;
    st = launch_tt_side_f32(sh, out, s, &handled);
    if (st != LRC_OK || handled) return st;
    return launch_chain<float>(sh, out, s);
}

lrc_status launch_tt_chain_f32tc(const TTShape& sh, float* out, cudaStream_t s) {
    return launch_chain<float>(sh, out, s, true);
}

lrc_status launch_tt_chain_f64(const TTShape& sh, double* out, cudaStream_t s) {
    return launch_chain<double>(sh, out, s);
}

// The binary64 chain with every product on the tensor cores (split_gemm.cu).
// Both operands of a product are cut into digits first: rows of Z, columns of
// the core (or of S).
lrc_status launch_tt_chain_f64_tc(const TTShape& sh, double* out, cudaStream_t s, bool* handled) {
    *handled = false;
    const int d = sh.d, c = plan_chain(sh).c;
    const double* const* G = reinterpret_cast<const double* const*>(sh.cores);
    struct Step {
        const double* A;
        const double* B;
        double* C;
        int64_t M, N, K;
        sg::Operand64 a, b;
        size_t oa, ob, oc;
    };
    std::vector<Step> steps;
    size_t off = 0, fix = 0;
    auto take = [&](size_t bytes) {
        const size_t o = off;
        off += round256(bytes);
        return o;
    };
    // A is M x K, B is K x N, both row-major (null: the step before's C on that side)
    auto add = [&](const double* A, const double* B, int64_t M, int64_t N, int64_t K, bool last) {
        Step t{A, B, nullptr, M, N, K, {}, {}, 0, 0, 0};
        t.a.rows = M;
        t.b.rows = N;
        t.a.K = t.b.K = K;
        t.oa = take(sg::operand_bytes(M, K));
        t.ob = take(sg::operand_bytes(N, K));
        fix = std::max(fix, sg::fix_bytes(M, N));
        t.oc = last ? 0 : take((size_t)M * (size_t)N * 8);
        steps.push_back(t);
    };
    int64_t P = sh.dims[0], Q = sh.dims[d - 1];
    for (int j = 1; j <= c - 1; ++j) {
        add(j == 1 ? G[0] : nullptr, G[j], P, sh.dims[j] * sh.ranks[j + 1], sh.ranks[j], false);
        P *= sh.dims[j];
    }
    const int left = (int)steps.size();
    for (int j = d - 2; j >= c; --j) {
        add(G[j], j == d - 2 ? G[d - 1] : nullptr, sh.ranks[j] * sh.dims[j], Q, sh.ranks[j + 1], false);
        Q *= sh.dims[j];
    }
    const int right = (int)steps.size();
    add(left ? nullptr : G[0], right > left ? nullptr : G[d - 1], P, Q, sh.ranks[c], true);
    const size_t o_f = take(fix), o_n = take(steps.size() * sizeof(int));      // list of one product after the other
    void* p = nullptr;
    lrc_status st = stream_workspace_try(s, off, &p);
    if (st != LRC_OK || !p) return st;
    *handled = true;
    unsigned char* ws = static_cast<unsigned char*>(p);
    int* counts = reinterpret_cast<int*>(ws + o_n);
    for (int i = 0; i < (int)steps.size(); ++i) {
        Step& t = steps[i];
        const bool last = i + 1 == (int)steps.size();
        const double* A = t.A ? t.A : (last ? steps[left - 1].C : steps[i - 1].C);
        const double* B = t.B ? t.B : (last ? steps[right - 1].C : steps[i - 1].C);
        t.C = last ? out : reinterpret_cast<double*>(ws + t.oc);
        sg::operand_carve(&t.a, ws + t.oa);
        sg::operand_carve(&t.b, ws + t.ob);
        t.a.src = sg::Src64{A, t.K, 1, nullptr, 0};
        t.b.src = sg::Src64{B, 1, t.N, nullptr, 0};
        const sg::Operand64* ops[2] = {&t.a, &t.b};
        const sg::Out64 o{t.C, t.N, 1, nullptr, nullptr};
        if ((st = sg::slice(ops, 2, counts, i == 0 ? (int)steps.size() : 0, s)) != LRC_OK) return st;
        const sg::Fix f{reinterpret_cast<int2*>(ws + o_f), counts + i};
        if ((st = sg::product(t.a, t.b, o, false, nullptr, f, s)) != LRC_OK) return st;
    }
    return LRC_OK;
}

// Where the digits' fixed cost (three launches a product, about 20 us a chain)
// pays: the FMA kernels take about 1 us per 1e6 flops (256^3, rank 34: 1.2e9
// flops, 1.1 ms -> 0.14 ms).  A tile of the product (128 x NT) costs about the
// same, 7 us of an SM, whatever its width and for all ranks up to 64, so the
// output product has to have enough to do in one: bond rank times NT from
// kTTDigitTile on.  Measured, digits / FMA kernels: 10^6 x 16 (NT = 16), rank 16
// 448 / 434 us, rank 4 440 / 115; 300^3 (NT = 64), ranks 8 183 / 424, 4 191 / 219,
// 2 288 / 115; 4096^2, rank 4 103 / 347, 2 151 / 195; 16384 x 8192, rank 1 543 /
// 295; 1000 x 1000 x 8, ranks 8 and 4 (NT = 16) 506 / 128.  Rows are numbered in 32 bits.
bool tt_chain_f64_tc_takes(const TTShape& sh) {
    constexpr double kTTDigitFlops = 4e7;
    constexpr int64_t kTTDigitTile = 192, kMost = (int64_t)1 << 31;
    const ChainPlan p = plan_chain(sh);
    if (p.flops < kTTDigitFlops) return false;
    int64_t P = 1, Q = 1;
    for (int j = 0; j < sh.d; ++j) {
        (j < p.c ? P : Q) *= sh.dims[j];
        // the products' other sides: core j's columns on the left, rows on the right
        if (j < p.c && sh.dims[j] * sh.ranks[j + 1] >= kMost) return false;
        if (j >= p.c && sh.ranks[j] * sh.dims[j] >= kMost) return false;
    }
    return P < kMost && Q < kMost && sh.ranks[p.c] * sg::product_tile(P, Q) >= kTTDigitTile;
}

bool tt_chain_saves(const TTShape& sh) { return plan_chain(sh).flops <= 0.8 * chain_flops(sh, sh.d - 1); }

}  // namespace lrc
