"""binary64 products on the tensor cores (split_gemm.cu; the apply, the TT
chain, the Gram matrices of eta): values cut into seven 9-bit digits, 28 exact
digit products, one rounding.

Integer data whose sums stay below 2^53 must come out exactly, whatever the
tiling; entries that the digits do not carry (sums of magnitudes far below the
rows' largest entries, infinities, NaN, extreme magnitudes) go through binary64
FMAs and must come out as they do."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from parity import packed, rel_fro

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


def run(lrc, dev, U, s, Vt, X):
    m, k = U.shape
    n, b = Vt.shape[1], X.shape[0]
    ops = [packed(lrc, a, "f64", dev) for a in (U, s, Vt, X)]
    Y = torch.full((b, m), float("nan"), dtype=torch.float64, device=dev)
    lrc.lrc_apply(*ops, Y, m, n, k, b, "f64")
    torch.cuda.synchronize()
    assert lrc.lrc_device_status() == 0
    return Y.cpu().numpy()


# tile edges of both orientations (128 rows by 16, 32, 48 or 64), reductions of
# one block, a partial chunk, several chunks with every drain period, odd sizes
SHAPES = [(129, 65, 33, 700), (1000, 64, 64, 128), (257, 1100, 300, 127), (4096, 17, 16, 200), (301, 2049, 40, 128),
          (64, 5000, 128, 17), (2051, 700, 97, 33), (127, 40000, 16, 129)]


@pytest.mark.parametrize("m,n,k,b", SHAPES)
def test_integers_are_exact(lrc, cuda, m, n, k, b):
    rng = np.random.default_rng(m + n)
    hi = max(2, int(2.0 ** (51 - 2 - np.log2(k) - 3 - np.log2(n) - 7)))     # the sums stay below 2^53
    X = rng.integers(-hi, hi + 1, (b, n)).astype(np.float64)
    Vt = rng.integers(-64, 65, (k, n)).astype(np.float64)
    U = rng.integers(-8, 9, (m, k)).astype(np.float64)
    s = rng.integers(-2, 3, k).astype(np.float64)
    want = ((X @ Vt.T) * s) @ U.T
    assert np.max(np.abs(want)) < 2.0 ** 53
    assert np.array_equal(run(lrc, cuda, U, s, Vt, X), want)


@pytest.mark.parametrize("m,n,k,b", SHAPES[:5])
def test_close_to_the_exact_product(lrc, cuda, m, n, k, b):
    """W and Y are each rounded once; digits and the classes left out add less:
    relative Frobenius error below 4 u against a product in extended precision."""
    f = W.random_factors(m, n, k, seed=7)
    X = W.gaussian((b, n), 8)
    got = run(lrc, cuda, f.U, f.s, f.Vt, X)
    L = np.longdouble
    want = ((X.astype(L) @ f.Vt.T.astype(L)) * f.s.astype(L)) @ f.U.T.astype(L)
    assert float(np.linalg.norm((got - want).astype(np.float64))) <= 4 * U64 * float(np.linalg.norm(want.astype(np.float64)))


def test_rows_the_digits_cannot_carry(lrc, cuda):
    m, n, k, b = 300, 777, 64, 130
    f = W.random_factors(m, n, k, seed=9)
    X = W.gaussian((b, n), 10)
    U, Vt = f.U.copy(), f.Vt.copy()
    rng = np.random.default_rng(11)
    X[3] *= 2.0 ** rng.integers(-200, 200, n)        # a wide row
    X[4] = 0.0
    X[5] *= 2.0 ** 600                               # beyond the digits' exponents
    U[17] *= 2.0 ** rng.integers(-90, 90, k)
    U[18] *= 2.0 ** -700
    Vt[2] *= 2.0 ** rng.integers(-90, 90, n)
    got = run(lrc, cuda, U, f.s, Vt, X)
    want = oracle.apply(U, f.s, Vt, X)
    bound = (np.abs(X) @ np.abs(Vt).T * np.abs(f.s)) @ np.abs(U).T
    assert np.all(np.abs(got - want) <= 2 * (n + k + 2) * U64 * bound)


@pytest.mark.parametrize("v", [np.inf, -np.inf, np.nan])
def test_nonfinite_values_spread_as_in_fma_sums(lrc, cuda, v):
    m, n, k, b = 200, 300, 64, 300
    f = W.random_factors(m, n, k, seed=12)
    X = W.gaussian((b, n), 13)
    U = f.U.copy()
    X[7, 5] = v
    U[9, 2] = v
    got = run(lrc, cuda, U, f.s, f.Vt, X)
    with np.errstate(invalid="ignore"):
        want = ((X @ f.Vt.T) * f.s) @ U.T
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(got[inf], want[inf])
    ok = np.isfinite(want)
    assert rel_fro(got[ok], want[ok]) <= 1e-14


def test_captured_call_and_repeat_are_the_same_bits(lrc, cuda):
    m, n, k, b = 600, 900, 48, 256
    f = W.random_factors(m, n, k, seed=14)
    X = W.gaussian((b, n), 15)
    ops = [packed(lrc, a, "f64", cuda) for a in (f.U, f.s, f.Vt, X)]
    Y = torch.empty((b, m), dtype=torch.float64, device=cuda)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        lrc.lrc_apply(*ops, Y, m, n, k, b, "f64", stream=st)
    torch.cuda.synchronize()
    want = Y.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        lrc.lrc_apply(*ops, Y, m, n, k, b, "f64", stream=st)
    Y.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(Y.view(torch.int64), want.view(torch.int64))


TT_SHAPES = [((130, 70, 90), (1, 20, 33, 1)), ((16, 16, 16, 16), (1, 16, 24, 16, 1)), ((300, 40, 129), (1, 7, 64, 1)),
             ((64, 2000), (1, 65, 1)), ((33, 17, 29, 31), (1, 30, 40, 20, 1))]


@pytest.mark.parametrize("dims,ranks", TT_SHAPES)
def test_tt_chain(lrc, cuda, dims, ranks):
    """Integer cores come out exactly; Gaussian ones within a few roundings of
    the chain's products of absolute values."""
    rng = np.random.default_rng(len(dims))
    d = len(dims)
    for integer in (True, False):
        cores = [rng.integers(-9, 10, (ranks[l], dims[l], ranks[l + 1])).astype(np.float64) if integer
                 else rng.standard_normal((ranks[l], dims[l], ranks[l + 1])) for l in range(d)]
        dev = [torch.from_numpy(c).to(cuda) for c in cores]
        out = torch.empty(int(np.prod(dims)), dtype=torch.float64, device=cuda)
        lrc.tt_reconstruct(dev, dims, ranks, "f64", out)
        torch.cuda.synchronize()
        assert lrc.lrc_device_status() == 0

        def chain(cs):
            z = cs[0].reshape(dims[0], -1)
            for c in cs[1:]:
                z = (z @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
            return z.reshape(-1)
        want = chain(cores)
        got = out.cpu().numpy()
        if integer:
            assert np.array_equal(got, want)
        else:
            bound = chain([np.abs(c) for c in cores])
            assert np.all(np.abs(got - want) <= (sum(ranks) + 2 * d) * U64 * bound)


@pytest.mark.parametrize("fmt", ["f16", "f32"])
@pytest.mark.parametrize("m,n,k", [(1500, 700, 65), (300, 2100, 130), (20000, 400, 32)])
def test_eta_through_digit_gram_matrices(lrc, cuda, fmt, m, n, k):
    f = W.random_factors(m, n, k, seed=21)
    wide = [packed(lrc, a, "f64", cuda) for a in (f.U, f.s, f.Vt)]
    low = [packed(lrc, a, fmt, cuda) for a in (f.U, f.s, f.Vt)]
    eta, norm = lrc.lrc_lowrank_eta(*wide, *low, fmt, m, n, k)
    L = np.longdouble
    Uh, sh, Vh = (oracle.rounded(a, fmt).astype(L) for a in (f.U, f.s, f.Vt))
    U, s, Vt = (a.astype(L) for a in (f.U, f.s, f.Vt))
    Pu, Pv = np.hstack([U - Uh, Uh]), np.vstack([Vt - Vh, Vh])
    M = np.zeros((2 * k, 2 * k), L)
    i = np.arange(k)
    M[i, i], M[i, k + i], M[k + i, i], M[k + i, k + i] = s, s, s, s - sh
    want = np.sqrt(np.sum((M.T @ (Pu.T @ Pu) @ M) * (Pv @ Pv.T)))
    assert abs(eta - float(want)) <= 1e-13 * float(want)
    assert abs(norm - float(np.linalg.norm(f.s))) <= 1e-12 * norm or k > min(m, n)


@pytest.mark.parametrize("m,n,k,b", [(4100, 600, 33, 700), (2050, 700, 40, 330), (1300, 2500, 70, 65), (130, 9000, 17, 65)])
def test_every_row_wide(lrc, cuda, m, n, k, b):
    """Entries over 60 binades in every row of V^T and U: digits over rows that
    hold mostly small entries, and what of them is recomputed, with partial tiles."""
    rng = np.random.default_rng(m)
    wide = lambda *s: rng.standard_normal(s) * 2.0 ** -rng.integers(0, 60, s)
    U, Vt, X, s = wide(m, k), wide(k, n), W.gaussian((b, n), 5), rng.uniform(0.5, 2.0, k)
    got = run(lrc, cuda, U, s, Vt, X)
    want = oracle.apply(U, s, Vt, X)
    bound = (np.abs(X) @ np.abs(Vt).T * np.abs(s)) @ np.abs(U).T
    assert np.all(np.abs(got - want) <= 2 * (n + k + 2) * U64 * bound)


@pytest.mark.parametrize("m,n,k", [(3000, 1700, 61), (16384, 8192, 144)])
def test_eta_of_wide_columns(lrc, cuda, m, n, k):
    """The Gram matrices of eta of columns over 40 binades (entries above the
    diagonal recomputed where the digits do not carry them, written both ways),
    against plain matrix products."""
    g = torch.Generator(device=cuda).manual_seed(m)
    rand = lambda *s: torch.randn(*s, generator=g, device=cuda, dtype=torch.float64)
    wide = lambda *s: rand(*s) * torch.exp2(-torch.randint(0, 40, s, generator=g, device=cuda).double())
    ld = lrc.lrc_packed_ld
    U = torch.zeros(m, ld(k), dtype=torch.float64, device=cuda)
    Vt = torch.zeros(k, ld(n), dtype=torch.float64, device=cuda)
    U[:, :k], Vt[:, :n] = wide(m, k), wide(k, n)
    s = rand(ld(k)).abs() + 0.1
    hats = [a.float() for a in (U, s, Vt)]
    eta, norm = lrc.lrc_lowrank_eta(U, s, Vt, *hats, "f32", m, n, k)
    # the trace forms with the rounding errors explicit, as in the header
    u, uh, v, vh = U[:, :k], hats[0][:, :k].double(), Vt[:, :n].T, hats[2][:, :n].double().T
    S, Sh = s[:k], hats[1][:k].double()
    P, Q = torch.cat([u - uh, uh], 1), torch.cat([v - vh, vh], 1)
    D = torch.diag
    M = torch.cat([torch.cat([D(S), D(S)], 1), torch.cat([D(S), D(S - Sh)], 1)], 0)
    Gu, Gv = P.T @ P, Q.T @ Q
    want = float(torch.sum((M.T @ Gu @ M) * Gv)) ** 0.5
    wnorm = float(torch.sum((D(S) @ (u.T @ u) @ D(S)) * (v.T @ v))) ** 0.5
    # a Gram entry has relative error (m + 2) u of its sum of magnitudes, and so
    # have eta^2's two factors; its terms (all of one size) nearly add up
    assert abs(eta - want) <= 8 * (m + n) * U64 * want
    assert abs(norm - wnorm) <= 8 * (m + n) * U64 * wnorm


@pytest.mark.parametrize("m,n,k,b,share,gap", [(300, 64, 600, 300, 0.5, 16), (257, 1000, 64, 300, 0.45, 18), (257, 1000, 64, 300, 0.27, 40),
                                               (130, 4099, 40, 200, 0.19, 59), (700, 1024, 33, 1000, 0.03, 70),
                                               (2050, 300, 130, 1100, 0.15, 25)])
def test_small_entries_that_are_all_that_counts(lrc, cuda, m, n, k, b, share, gap):
    """A share of every row's entries lies 2^-gap below the others, and the other
    operand is zero beside them: digits below the large entries hold little or
    nothing of the result.  Both products, against the sums of magnitudes."""
    rng = np.random.default_rng(gap)

    def scaled(rows, cols):
        small = rng.permutation(cols) < max(1, int(share * cols))
        return rng.standard_normal((rows, cols)) * np.where(small, 2.0 ** -gap, 1.0), small
    Vt, small = scaled(k, n)
    X = rng.standard_normal((b, n)) * small
    U, small_k = scaled(m, k)
    s = np.where(small_k, rng.uniform(0.5, 2.0, k), 0.0)
    for args in ((rng.standard_normal((m, k)), np.ones(k), Vt, X), (U, s, rng.standard_normal((k, n)), rng.standard_normal((b, n))),
                 (U, s, Vt, X)):
        want = oracle.apply(*args)
        u, t, v, x = (np.abs(a) for a in args)
        bound = ((x @ v.T) * t) @ u.T
        assert np.all(np.abs(run(lrc, cuda, *args) - want) <= 2 * (n + k + 2) * U64 * bound)


@pytest.mark.parametrize("m,n,k,b", [(70, 4096, 64, 64), (301, 600, 130, 2003), (4100, 100, 33, 300), (3001, 95, 97, 171)])
def test_every_entry_listed(lrc, cuda, m, n, k, b):
    """Disjoint large entries in every row of both products: blocks and single
    entries, few and many, partial blocks at both edges, short and long sums."""
    rng = np.random.default_rng(n)
    even, even_k = np.arange(n) % 2 == 0, np.arange(k) % 2 == 0
    X = rng.standard_normal((b, n)) * even
    Vt = rng.standard_normal((k, n)) * np.where(even, 2.0 ** -30, 1.0) * even_k[:, None]
    U = rng.standard_normal((m, k)) * np.where(even_k, 2.0 ** -30, 1.0)
    s = rng.uniform(0.5, 2.0, k)
    want = oracle.apply(U, s, Vt, X)
    bound = ((np.abs(X) @ np.abs(Vt).T) * s) @ np.abs(U).T
    assert np.all(np.abs(run(lrc, cuda, U, s, Vt, X) - want) <= 2 * (n + k + 2) * U64 * bound)


def test_unit_and_zero_queries(lrc, cuda):
    """One entry a query: Y is a column of A, whatever the size of its entries;
    zero queries make zeros beside an infinite factor entry that they meet NaN."""
    m, n, k, b = 500, 1100, 64, 400
    f = W.random_factors(m, n, k, seed=31)
    X = np.zeros((b, n))
    X[np.arange(b), (np.arange(b) * 7) % n] = 3.0
    X[5] = X[77] = 0.0
    got = run(lrc, cuda, f.U, f.s, f.Vt, X)
    want = oracle.apply(f.U, f.s, f.Vt, X)
    bound = ((np.abs(X) @ np.abs(f.Vt).T) * f.s) @ np.abs(f.U).T
    assert np.all(np.abs(got - want) <= 2 * (k + 4) * U64 * bound)
    U = f.U.copy()
    U[9, 2] = np.inf
    got = run(lrc, cuda, U, f.s, f.Vt, X)
    assert np.all(np.isnan(got[[5, 77], 9])) and np.all(got[5, :9] == 0) and np.all(got[77, 10:] == 0)


def test_digits_at_their_limits(lrc, cuda):
    """Constant rows of the value whose digits are 65, -256, ..., -256: what the
    classes left out add has one sign and its largest size, below 2^-57 of the
    power of two above the entries, squared, a term."""
    n, k, b, m = 2048, 128, 64, 64
    v = (65 * 2 ** 54 - sum(256 << (54 - 9 * i) for i in range(1, 7))) / 2.0 ** 61
    got = run(lrc, cuda, np.full((m, k), v), np.ones(k), np.full((k, n), v), np.full((b, n), v))
    L = np.longdouble
    want = L(v) ** 3 * n * k
    assert np.all(np.abs(got.astype(L) - want) <= (2 * U64 + 2 * 2.0 ** -57 / v ** 2) * want)


@pytest.mark.parametrize("dims,ranks", TT_SHAPES)
def test_tt_chain_of_blocks_of_different_size(lrc, cuda, dims, ranks):
    """Half of every bond's slices 2^-20 ... 2^-60 below the others on one side,
    and zero or larger on the other."""
    rng = np.random.default_rng(8)
    d = len(dims)
    cores = [rng.standard_normal((ranks[l], dims[l], ranks[l + 1])) for l in range(d)]
    for l in range(1, d):
        half = np.arange(ranks[l]) % 2 == 0
        cores[l - 1] = cores[l - 1] * np.where(half, 2.0 ** -(20 * l), 1.0)
        cores[l] = cores[l] * np.where(half, 1.0, 0.0)[:, None, None] if l % 2 else cores[l] * np.where(half, 1.0, 2.0 ** -30)[:, None, None]
    dev = [torch.from_numpy(np.ascontiguousarray(c)).to(cuda) for c in cores]
    out = torch.empty(int(np.prod(dims)), dtype=torch.float64, device=cuda)
    lrc.tt_reconstruct(dev, dims, ranks, "f64", out)
    torch.cuda.synchronize()

    def chain(cs):
        z = cs[0].reshape(dims[0], -1)
        for c in cs[1:]:
            z = (z @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
        return z.reshape(-1)
    bound = chain([np.abs(c) for c in cores])
    assert np.all(np.abs(out.cpu().numpy() - chain(cores)) <= (sum(ranks) + 2 * d) * U64 * bound)


@pytest.mark.parametrize("dims,ranks", [((3000, 2500), (1, 3, 1)), ((3000, 2500), (1, 2, 1)), ((200000, 16), (1, 11, 1)),
                                        ((200000, 16), (1, 12, 1)), ((16, 90000), (1, 16, 1)), ((1500, 70, 90), (1, 4, 3, 1)),
                                        ((1500, 70, 48), (1, 8, 4, 1))])
def test_tt_low_ranks_and_thin_sides(lrc, cuda, dims, ranks):
    """Both sides of the rule on bond rank times tile width."""
    g = torch.Generator(device=cuda).manual_seed(6)
    d = len(dims)
    cores = [torch.randn(ranks[l], dims[l], ranks[l + 1], generator=g, device=cuda, dtype=torch.float64) for l in range(d)]
    out = torch.empty(int(np.prod(dims)), dtype=torch.float64, device=cuda)
    lrc.tt_reconstruct(cores, dims, ranks, "f64", out)

    def full(cs):
        z = cs[0].reshape(dims[0], -1)
        for c in cs[1:]:
            z = (z @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
        return z.reshape(-1)
    want, bound = full(cores), full([c.abs() for c in cores])
    # a few roundings here, the reference's sums
    assert torch.all((out - want).abs() <= 2 * (sum(ranks) + 2 * d) * U64 * bound)


@pytest.mark.parametrize("m,n,k,b", [(300, 1100, 64, 1100), (200, 5000, 40, 700), (257, 300, 33, 2100)])
def test_identity_and_sign_queries(lrc, cuda, m, n, k, b):
    """Rows with first digits only lose nothing but the other row's rounding: the
    identity gives the rows of V (to u of each), a few signs u of their sums."""
    rng = np.random.default_rng(n)
    Vt = rng.standard_normal((k, n)) * 2.0 ** -rng.integers(0, 12, (k, n))
    U = np.eye(m, k)
    X = np.zeros((b, n))
    X[np.arange(b), np.arange(b) % n] = 1.0
    few = np.arange(b) % 3 == 0
    X[few] += (rng.random((few.sum(), n)) < 5 / n) * rng.choice([-1.0, 1.0, 3.0], (few.sum(), n))
    got = run(lrc, cuda, U, np.ones(k), Vt, X)[:, :min(m, k)]
    want = (X @ Vt.T)[:, :min(m, k)]
    terms = np.count_nonzero(X, axis=1)[:, None]
    assert np.all(np.abs(got - want) <= (2 * terms + 2) * U64 * (np.abs(X) @ np.abs(Vt).T)[:, :min(m, k)])


@pytest.mark.parametrize("m,n,k", [(3000, 1700, 61), (20000, 900, 40), (9000, 8192, 144)])
def test_eta_of_columns_outside_the_digits_exponents(lrc, cuda, m, n, k):
    """Every entry of one Gram matrix (upper tiles, written both ways) formed by
    FMAs: the same eta as of the factors scaled into the digits' range."""
    g = torch.Generator(device=cuda).manual_seed(k)
    rand = lambda *s: torch.randn(*s, generator=g, device=cuda, dtype=torch.float64)
    ld = lrc.lrc_packed_ld
    U, Vt = rand(m, ld(k)), rand(k, ld(n))
    s = rand(ld(k)).abs() + 0.1
    hats = [a * (1 + 1e-6 * rand(*a.shape)) for a in (U, s, Vt)]
    eta, norm = lrc.lrc_lowrank_eta(U, s, Vt, *hats, "f64", m, n, k)
    down, up = 2.0 ** -485, 2.0 ** 400
    e2, n2 = lrc.lrc_lowrank_eta(U * down, s * up, Vt, hats[0] * down, hats[1] * up, hats[2], "f64", m, n, k)
    assert lrc.lrc_device_status() == 0
    # m terms a Gram entry, each way of summing within (m + 2) u of its magnitudes
    assert abs(e2 / (down * up) - eta) <= 4 * (m + n) * U64 * eta
    assert abs(n2 / (down * up) - norm) <= 4 * (m + n) * U64 * norm
