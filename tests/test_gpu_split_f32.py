"""binary32 products on the tensor cores (split_gemm32.cu): three bfloat16
parts of every value, six products of parts.

Integer data whose sums stay below 2^24 must come out exactly, whatever the
tiling; rows with entries that the parts cannot carry go through binary32 FMAs
and must come out as they do."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from parity import packed

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


def run(lrc, dev, U, s, Vt, X, fmt="f32"):
    m, k = U.shape
    n, b = Vt.shape[1], X.shape[0]
    ops = [packed(lrc, a, fmt, dev) for a in (U, s, Vt, X)]
    Y = torch.full((b, m), float("nan"), dtype=torch.float32, device=dev)
    lrc.lrc_apply(*ops, Y, m, n, k, b, fmt)
    torch.cuda.synchronize()
    assert lrc.lrc_device_status() == 0
    return Y.double().cpu().numpy()


# row and column tiles' edges, output rows with and without a 16-byte pitch,
# reductions of one block, a partial chunk, past one drain of the lower products
SHAPES = [(300, 7777, 33, 520), (129, 4100, 65, 380), (4097, 4096, 16, 900), (1000, 1030, 129, 900), (256, 16384, 40, 200),
          (2050, 5000, 17, 1025), (515, 4099, 272, 128)]


@pytest.mark.parametrize("m,n,k,b", SHAPES)
def test_integers_are_exact(lrc, cuda, m, n, k, b):
    rng = np.random.default_rng(m + n)
    X = rng.integers(-1, 2, (b, n)).astype(np.float64) * (rng.random((b, n)) < 0.05) * 17
    Vt = rng.integers(-3, 4, (k, n)).astype(np.float64)
    U = rng.integers(-2, 3, (m, k)).astype(np.float64) * (rng.random((m, k)) < 0.2)
    s = rng.integers(0, 2, k).astype(np.float64)
    W1 = X @ Vt.T
    want = (W1 * s) @ U.T
    assert max(np.max(np.abs(X) @ np.abs(Vt).T), np.max((np.abs(W1) * s) @ np.abs(U).T)) < 2.0 ** 24
    assert np.array_equal(run(lrc, cuda, U, s, Vt, X), want)


@pytest.mark.parametrize("fmt", ["f32", "f32tc"])
@pytest.mark.parametrize("m,n,k,b", SHAPES)
def test_no_further_from_the_exact_product_than_fma_sums(lrc, cuda, m, n, k, b, fmt):
    """A sum of K binary32 FMAs in blocks of 1024 is off by about 0.2 sqrt(1024)
    roundings of random sign; allow 8 u relative Frobenius (n + k terms)."""
    f = W.random_factors(m, n, k, seed=7)
    X = W.gaussian((b, n), 8)
    U, s, Vt, X = (oracle.rounded(a, "f32") for a in (f.U, f.s, f.Vt, X))
    want = ((X @ Vt.T) * s) @ U.T
    got = run(lrc, cuda, U, s, Vt, X, fmt)
    assert np.linalg.norm(got - want) <= 8 * U32 * np.linalg.norm(want)


def test_rows_the_parts_cannot_carry(lrc, cuda):
    m, n, k, b = 300, 4100, 64, 520
    f = W.random_factors(m, n, k, seed=9)
    X = W.gaussian((b, n), 10)
    U, Vt = f.U.copy(), f.Vt.copy()
    X[3] *= 2.0 ** -110
    X[4] = 0.0
    X[5, 7] = 2.0 ** 127
    X[6, 9] = 2.0 ** -140
    U[17, 3] = 2.0 ** -130
    Vt[2] *= 2.0 ** -20
    U, s, Vt, X = (oracle.rounded(a, "f32") for a in (U, f.s, Vt, X))
    got = run(lrc, cuda, U, s, Vt, X)
    want = oracle.apply(U, s, Vt, X)
    bound = ((np.abs(X) @ np.abs(Vt).T) * np.abs(s)) @ np.abs(U).T
    assert np.all(np.abs(got - want) <= 64 * U32 * bound + 2.0 ** -140)


@pytest.mark.parametrize("v", [np.inf, -np.inf, np.nan, 3.0e38])
def test_nonfinite_values_spread_as_in_fma_sums(lrc, cuda, v):
    m, n, k, b = 200, 4300, 64, 400
    f = W.random_factors(m, n, k, seed=12)
    X = W.gaussian((b, n), 13)
    U = f.U.copy()
    X[7, 5] = v
    U[9, 2] = v
    U, s, Vt, X = (oracle.rounded(a, "f32") for a in (U, f.s, f.Vt, X))
    got = run(lrc, cuda, U, s, Vt, X)
    with np.errstate(invalid="ignore", over="ignore"):
        want = (((X @ Vt.T).astype(np.float32) * s.astype(np.float32)).astype(np.float64) @ U.T).astype(np.float32).astype(np.float64)
    if np.isfinite(v):          # sums near the end of the range: only their neighbours are compared
        keep = np.ones(b, bool)
        keep[7] = False
        ok = np.isfinite(want) & keep[:, None]
    else:
        assert np.array_equal(np.isnan(got), np.isnan(want))
        inf = np.isinf(want)
        assert np.array_equal(got[inf], want[inf])
        ok = np.isfinite(want)
    ok[:, 9] = False
    assert np.linalg.norm(got[ok] - want[ok]) <= 8 * U32 * np.linalg.norm(want[ok])


def test_repeat_is_the_same_bits(lrc, cuda):
    m, n, k, b = 700, 5000, 48, 500
    f = W.random_factors(m, n, k, seed=14)
    X = W.gaussian((b, n), 15)
    assert np.array_equal(run(lrc, cuda, f.U, f.s, f.Vt, X), run(lrc, cuda, f.U, f.s, f.Vt, X))


def chain(cores, dims):
    z = cores[0].reshape(dims[0], -1)
    with np.errstate(invalid="ignore", over="ignore"):
        for c in cores[1:]:
            z = (z @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
    return z.reshape(-1)


# small cores (the side kernel's images), and an output product large enough for
# the parts of split_gemm32.cu, with and without a 16-byte row pitch
TT_SHAPES = [((16, 16, 16, 16), (1, 16, 26, 16, 1)), ((33, 17, 29, 31), (1, 30, 40, 20, 1)), ((64, 70, 60), (1, 12, 60, 1)),
             ((400, 100, 1000), (1, 9, 36, 1)), ((300, 130, 1001), (1, 40, 33, 1))]


@pytest.mark.parametrize("fmt,bad", [("f32", None), ("f32tc", None), ("f32", np.inf), ("f32", np.nan),
                                     ("f32", -3.4028234e38)])
@pytest.mark.parametrize("dims,ranks", TT_SHAPES)
def test_tt(lrc, cuda, dims, ranks, fmt, bad):
    """An infinity among positive cores makes its entries infinite, a NaN NaN,
    whatever the order of the chain."""
    rng = np.random.default_rng(5)
    d = len(dims)
    cores = [oracle.rounded(rng.standard_normal((ranks[l], dims[l], ranks[l + 1])), "f32") for l in range(d)]
    if bad is not None:
        cores = [oracle.rounded(np.abs(c) * 1e-3 + 1e-6, "f32") for c in cores]
        cores[0][0, 3, 1] = bad
        cores[-1][2, 5, 0] = bad if abs(bad) == np.inf else cores[-1][2, 5, 0]
    dev = [torch.from_numpy(c).float().to(cuda) for c in cores]
    out = torch.empty(int(np.prod(dims)), dtype=torch.float32, device=cuda)
    lrc.tt_reconstruct(dev, dims, ranks, fmt, out)
    torch.cuda.synchronize()
    assert lrc.lrc_device_status() == 0
    want, got = chain(cores, dims), out.double().cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want)
    assert np.array_equal(got[inf], want[inf])
    ok = np.isfinite(want)
    # roundings of the chain's sums, relative to the sums of magnitudes
    bound = chain([np.where(np.isfinite(c), np.abs(c), 1.0) for c in cores], dims)
    assert np.all(np.abs(got[ok] - want[ok]) <= 8 * np.sqrt(max(ranks)) * U32 * bound[ok] * d)


@pytest.mark.parametrize("m,n,k,b", [(4100, 600, 136, 1100), (2050, 8300, 40, 520), (12000, 9000, 33, 250)])
def test_every_row_recomputed(lrc, cuda, m, n, k, b):
    """Entries of 1e-34 in every row of V^T and U, whose unscaled parts would fall
    below bfloat16's range."""
    rng = np.random.default_rng(m)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    small = lambda a: f32(np.where(np.arange(a.shape[1]) % 5 == 0, a * 1e-34, a))
    U, Vt = small(rng.standard_normal((m, k))), small(rng.standard_normal((k, n)))
    X, s = f32(rng.standard_normal((b, n))), f32(rng.uniform(0.5, 2.0, k))
    got = run(lrc, cuda, U, s, Vt, X)
    want = ((X @ Vt.T) * s) @ U.T
    bound = (np.abs(X) @ np.abs(Vt).T * s) @ np.abs(U).T
    # sums of at most 1024 terms and of their sums, two products, one scaling
    assert np.all(np.abs(got - want) <= 2 * (min(n, 1024) + n / 1024 + k + 4) * U32 * bound)


@pytest.mark.parametrize("fmt", ["f32", "f32tc"])
def test_products_near_the_ends_of_the_range(lrc, cuda, fmt):
    """Products beyond binary32's range are infinite (not a NaN from parts that
    overflow apart), those inside it finite, and those of entries down to the
    smallest subnormal numbers as close as FMA sums."""
    m, n, k, b = 300, 5000, 64, 600
    f32 = lambda a: np.asarray(a, np.float64).astype(np.float32).astype(np.float64)
    rng = np.random.default_rng(17)
    X, Vt, U = f32(rng.standard_normal((b, n))), f32(rng.standard_normal((k, n))), f32(rng.standard_normal((m, k)))
    s = np.ones(k)
    X[3] = X[4] = X[5] = X[6] = 0.0
    X[3, 9], Vt[7, 9] = f32(1.99 * 2.0 ** 70), f32(1.99 * 2.0 ** 70)
    X[4, 11], Vt[8, 11] = f32(1.998 * 2.0 ** 64), f32(0.9989 * 2.0 ** 63)          # 0.998 2^128
    X[5, 13], Vt[9, 13] = 2.0 ** -60, f32(1.7 * 2.0 ** -85)
    X[6] = f32(rng.standard_normal(n) * 2.0 ** -rng.integers(100, 149, n))
    U[:, 7:10] = 0.0
    U[10, 7], U[11, 8], U[12, 9] = 1.0, f32(0.9), 1.0
    U[13] = f32(rng.standard_normal(k) * 2.0 ** -rng.integers(100, 149, k))
    got = run(lrc, cuda, U, s, Vt, X, fmt)
    assert got[3, 10] == np.inf and np.isnan(got[3, 9])          # (0 times infinity)
    W1 = X @ Vt.T
    W1 = f32(np.where(np.abs(W1) < 2.0 ** 128, W1, np.inf))
    rows = np.arange(b) != 3
    want, bound = W1[rows] @ U.T, (np.abs(X[rows]) @ np.abs(Vt).T) @ np.abs(U).T
    assert np.isfinite(got[4, 11]) and np.isfinite(want).all()
    assert np.all(np.abs(got[rows] - want) <= 64 * U32 * bound + k * 2.0 ** -149)


@pytest.mark.parametrize("m,n,k,b", [(4100, 600, 136, 1100), (2050, 8300, 40, 520), (12000, 9000, 33, 250)])
def test_every_row_above_the_limit(lrc, cuda, m, n, k, b):
    """Entries above the parts' limit in every row of V^T and U: both products in
    the tiles that the repair takes for many and few entries."""
    rng = np.random.default_rng(m)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    large = lambda a: f32(np.where(np.arange(a.shape[1]) % 5 == 0, a * 2.0 ** 40, a))
    U, Vt = large(rng.standard_normal((m, k))), large(rng.standard_normal((k, n)))
    X, s = f32(rng.standard_normal((b, n))), f32(rng.uniform(0.5, 2.0, k))
    got = run(lrc, cuda, U, s, Vt, X)
    want = ((X @ Vt.T) * s) @ U.T
    bound = (np.abs(X) @ np.abs(Vt).T * s) @ np.abs(U).T
    # sums of at most 1024 terms and of their sums, two products, one scaling
    assert np.all(np.abs(got - want) <= 2 * (min(n, 1024) + n / 1024 + k + 4) * U32 * bound)


@pytest.mark.parametrize("dims,ranks", [((300, 200), (1, 20, 1)), ((4096, 4096), (1, 48, 1))])
def test_two_cores_captured_without_workspace(lrc, cuda, dims, ranks):
    """A two-core binary32 chain needs no workspace: as the first call on its
    stream it can be captured, and gives what FMA sums give."""
    g = torch.Generator(device=cuda).manual_seed(3)
    cores = [torch.randn(ranks[l], dims[l], ranks[l + 1], generator=g, device=cuda) for l in range(2)]
    out = torch.zeros(dims, device=cuda)
    torch.cuda.synchronize()
    lrc.lrc_shutdown()                      # no stream has a workspace
    st = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        lrc.tt_reconstruct(cores, dims, ranks, "f32", out, stream=st)
    graph.replay()
    torch.cuda.synchronize()
    a, b = (c.reshape(-1, c.shape[2]).double() if l == 0 else c.reshape(c.shape[0], -1).double() for l, c in enumerate(cores))
    assert torch.all((out.double() - a @ b).abs() <= (ranks[1] + 2) * U32 * (a.abs() @ b.abs()))


def test_tt_rows_of_very_different_size(lrc, cuda):
    """Rows of 2^18 down to 2^-124 in every group of 32, on either side: a row times
    a unit column comes out as it is; and entries near both ends of the range."""
    m, q = 96, 160
    rng = np.random.default_rng(2)
    f32 = lambda a: a.astype(np.float32)
    scale = 2.0 ** np.floor(18 - 142 / 31 * (np.arange(m) % 32))
    for flip in (False, True):
        A = f32(np.stack([rng.standard_normal(m) * scale, rng.standard_normal(m) * 1e-3], 1))
        B = np.zeros((2, q), np.float32)
        B[0] = 2.0 ** (np.arange(q) % 3)
        if flip:
            A, B = np.ascontiguousarray(B.T), np.ascontiguousarray(A.T)
        dims = (A.shape[0], B.shape[1])
        out = torch.empty(dims, device=cuda)
        cores = [torch.from_numpy(A)[None].to(cuda), torch.from_numpy(B)[:, :, None].to(cuda)]
        lrc.tt_reconstruct(cores, dims, (1, 2, 1), "f32", out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), f32(A.astype(np.float64) @ B.astype(np.float64)))
    A = f32(rng.uniform(1, 2, (40, 2)) * np.array([2.0 ** 126, 0.0]))
    B = f32(rng.uniform(1, 2, (2, 40)) * 2.0 ** -np.linspace(0, 140, 40)[None, :])
    out = torch.empty((40, 40), device=cuda)
    lrc.tt_reconstruct([torch.from_numpy(A)[None].to(cuda), torch.from_numpy(B)[:, :, None].to(cuda)], (40, 40), (1, 2, 1), "f32", out)
    with np.errstate(over="ignore"):
        want = f32(A.astype(np.float64) @ B.astype(np.float64)).astype(np.float64)
    got = out.double().cpu().numpy()
    assert np.array_equal(np.isinf(got), np.isinf(want))
    ok = np.isfinite(want)
    assert np.all(np.abs(got[ok] - want[ok]) <= 4 * U32 * np.abs(want[ok]))


@pytest.mark.parametrize("fmt", ["f32", "f32tc"])
@pytest.mark.parametrize("dims,ranks", [((20000, 16), (1, 16, 1)), ((16, 20001), (1, 5, 1)), ((200, 100, 8), (1, 8, 4, 1)),
                                        ((9600, 96), (1, 16, 1)), ((9600, 97), (1, 16, 1)), ((8, 50, 60, 5), (1, 8, 20, 5, 1)),
                                        ((2100, 500), (1, 17, 1)), ((700, 1500), (1, 64, 1))])
def test_tt_thin_sides(lrc, cuda, dims, ranks, fmt):
    """Both sides of the rule that sends thin tensors past the images."""
    g = torch.Generator(device=cuda).manual_seed(5)
    d = len(dims)
    cores = [torch.randn(ranks[l], dims[l], ranks[l + 1], generator=g, device=cuda) for l in range(d)]
    out = torch.empty(int(np.prod(dims)), device=cuda)
    lrc.tt_reconstruct(cores, dims, ranks, fmt, out)

    def full(cs):
        z = cs[0].reshape(dims[0], -1)
        for c in cs[1:]:
            z = (z @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[2])
        return z.reshape(-1)
    want, bound = full([c.double() for c in cores]), full([c.double().abs() for c in cores])
    # f32tc: 22 bits an operand of the largest of 32 rows, four times a rounding each
    assert torch.all((out.double() - want).abs() <= (sum(ranks) + 2 * d + (64 if fmt == "f32tc" else 0)) * U32 * bound + (
        8 * U32 * bound.max() if fmt == "f32tc" else 0))
