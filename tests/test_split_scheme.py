"""The arithmetic scheme of the FP32 tensor-core variant (LRC_F32_TC),
emulated in numpy on the CPU: binary32 values scaled by a power of two per
group (largest magnitude into [2^14, 2^15)) and split into binary16 parts
hi = fp16(x), lo = fp16(x - hi) keep about 22 bits of the group's scale,
and the three products W_hi U_hi + W_lo U_hi + W_hi U_lo stay within the
binary32 tolerance of the exact product."""
import numpy as np


def group_exp(maxabs):
    if not (maxabs > 0) or not np.isfinite(maxabs):
        return 0
    e = 14 - int(np.floor(np.log2(np.float32(maxabs))))
    return int(np.clip(e, -60, 60))


def split(x32, group_rows):
    """Parts of a binary32 matrix, scaled per group of rows (1 = per row)."""
    hi = np.empty(x32.shape, np.float16)
    lo = np.empty(x32.shape, np.float16)
    ex = np.empty(x32.shape[0], np.int64)
    for r0 in range(0, x32.shape[0], group_rows):
        g = x32[r0:r0 + group_rows]
        e = group_exp(float(np.max(np.abs(g))))
        y = (g * np.float32(2.0 ** e)).astype(np.float32)          # exact: a power of two
        h = y.astype(np.float16)
        l = (y - h.astype(np.float32)).astype(np.float16)          # residual exact in binary32
        hi[r0:r0 + group_rows], lo[r0:r0 + group_rows], ex[r0:r0 + group_rows] = h, l, e
    return hi, lo, ex


def test_parts_keep_22_bits_of_the_group_scale():
    rng = np.random.default_rng(5)
    x = (rng.standard_normal((256, 96)) * np.exp2(rng.integers(-40, 40, size=(256, 1)))).astype(np.float32)
    for group in (1, 32):
        hi, lo, ex = split(x, group)
        back = (hi.astype(np.float64) + lo.astype(np.float64)) * np.exp2(-ex.astype(np.float64))[:, None]
        for r0 in range(0, 256, group):
            g = slice(r0, r0 + group)
            scale = np.max(np.abs(x[g].astype(np.float64)))
            assert np.max(np.abs(back[g] - x[g])) <= 2.0 ** -22 * scale


def test_scaling_is_what_keeps_the_bits():
    """A group of magnitude about 1e-3 split without the power-of-two scale
    leaves lo among the binary16 subnormals (absolute step 2^-24) and keeps
    only about 17 bits of the group's scale; scaled, it keeps 22."""
    rng = np.random.default_rng(7)
    x = (rng.standard_normal((32, 64)) * 1e-3).astype(np.float32)
    scale = np.max(np.abs(x.astype(np.float64)))
    h = x.astype(np.float16)
    l = (x - h.astype(np.float32)).astype(np.float16)
    err_plain = np.max(np.abs(h.astype(np.float64) + l.astype(np.float64) - x))
    hi, lo, ex = split(x, 32)
    back = (hi.astype(np.float64) + lo.astype(np.float64)) * np.exp2(-float(ex[0]))
    err_scaled = np.max(np.abs(back - x))
    assert err_plain > 2.0 ** -18 * scale
    assert err_scaled <= 2.0 ** -22 * scale
    assert err_plain >= 16 * err_scaled


def test_three_products_meet_the_binary32_tolerance():
    rng = np.random.default_rng(6)
    b, m, k = 64, 200, 136
    W = (rng.standard_normal((b, k)) * np.exp2(rng.integers(-20, 20, size=(b, 1)))).astype(np.float32)
    U = rng.standard_normal((m, k)).astype(np.float32)
    Wh, Wl, ew = split(W, 1)
    Uh, Ul, eu = split(U, 32)
    f = lambda a: a.astype(np.float64)                                 # noqa: E731
    Y = (f(Wh) @ f(Uh).T + f(Wl) @ f(Uh).T + f(Wh) @ f(Ul).T)
    Y *= np.exp2(-ew.astype(np.float64))[:, None] * np.exp2(-eu.astype(np.float64))[None, :]
    exact = f(W) @ f(U).T
    rel = np.linalg.norm(Y - exact, axis=1) / np.linalg.norm(exact, axis=1)
    assert rel.max() <= 1e-6, rel.max()
    # the dropped term W_lo U_lo is below 2^-22 of the product's scale
    assert np.max(np.abs(f(Wl) @ f(Ul).T)) <= 2.0 ** -22 * np.max(np.abs(f(Wh) @ f(Uh).T)) * 4


# ---- binary64 from seven 9-bit digits (split_gemm.cu)

def digits(x):
    """Digits (rows, 7, columns) of rows of binary64 numbers, as Python integers,
    and the exponents of the power of two above each row's largest entry."""
    top = np.array([np.frexp(np.max(np.abs(r)))[1] for r in x])
    v = np.array([[int(np.rint(np.ldexp(e, 61 - t))) for e in r] for r, t in zip(x, top)], dtype=object)
    bias = sum(256 << (54 - 9 * i) for i in range(1, 7))
    t = v + bias
    d = [t >> 54] + [((t >> (54 - 9 * i)) & 511) - 256 for i in range(1, 7)]
    return np.stack(d, 1), top


def check_unlisted(a, b, far_off=False):
    """Entries whose first digits' sum of magnitudes reaches 2^9, or 2^5 where a row
    has first digits only, are within K 2^-50 of the exact sum of magnitudes (then
    within 2^-52 for every term that is not zero); the others are left to FMAs."""
    K = a.shape[1]
    (da, ta), (db, tb) = digits(a), digits(b)
    kept = sum((da[:, i] @ db[:, j].T) * (1 << (9 * (6 - i - j))) for i in range(7) for j in range(7 - i))
    est = abs(da[:, 0]) @ abs(db[:, 0]).T
    ia, ib = (np.array([[int(np.ldexp(e, 61 - t + 200)) for e in r] for r, t in zip(x, top)], dtype=object)
              for x, top in ((a, ta), (b, tb)))
    exact, mags = ia @ ib.T, abs(ia) @ abs(ib).T              # in units of 2^-400 of the digits' square
    err = abs(kept * (1 << 54) * (1 << 400) - exact)
    short = np.logical_or.outer(np.all(da[:, 1:] == 0, (1, 2)), np.all(db[:, 1:] == 0, (1, 2)))
    on = np.asarray(est >= np.where(short, 32, 512), bool)
    assert np.all(err[on] * (1 << 50) <= K * mags[on])
    terms = np.asarray(ia != 0, int) @ np.asarray(ib != 0, int).T
    assert np.all(err[on & short] * (1 << 52) <= terms[on & short] * mags[on & short])
    if far_off:        # what the limit is for: digits alone would miss the FMA bound
        assert np.any(err[~on] * (1 << 53) > 64 * K * mags[~on])
    return on


def test_digits_carry_what_the_estimate_passes():
    rng = np.random.default_rng(3)
    g = lambda *s: rng.standard_normal(s)
    assert check_unlisted(g(12, 64), g(9, 64)).all()
    assert check_unlisted(g(12, 40) * np.arange(1, 41) ** -0.75, g(9, 40) * np.arange(1, 41) ** -0.75).all()
    limits = np.full((2, 48), (65 * 2 ** 54 - sum(256 << (54 - 9 * i) for i in range(1, 7))) / 2.0 ** 61)
    assert check_unlisted(limits, limits).all()
    for gap in (12, 20, 40, 70):
        small = np.arange(64) % 4 == 0
        a = g(12, 64) * np.where(small, 2.0 ** -gap, 1.0)
        check_unlisted(a, np.vstack([g(5, 64) * small, g(4, 64)]), gap >= 20)
    on = check_unlisted(np.vstack([np.eye(20, 64), rng.integers(-3, 4, (9, 64)).astype(float)]), g(9, 64))
    assert 0.9 < on[:20].mean() < 1 and on[20:].all()
    check_unlisted(g(12, 64) * 2.0 ** -rng.integers(0, 60, (12, 64)), g(9, 64) * 2.0 ** -rng.integers(0, 60, (9, 64)))
