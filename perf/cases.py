"""What this framework's speed is judged on: calls that a program makes of it.

A program holds the factors of a truncated SVD (or the cores of a Tensor
Train) in one of the storage formats and uses them through the package's
entry points:

* it applies them to batches of queries -- one or a few queries at a time when
  it serves, thousands when it processes a data set -- alone or for a set of
  matrices at once;
* it reconstructs a dense tensor from its cores;
* it stores binary64 factors or cores in a narrower format and measures the
  perturbation eta that the accuracy certificate needs, by the fused route or
  by the dense one.

Sizes, ranks and spectra are those of the benchmark's workloads and of the
tests; `draw` spreads over the same ranges, odd sizes included.
"""
import math

import torch

import paper_2607_12969_gb300 as lrc

DEV = "cuda:0"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest apply: factors and queries of one small matrix, bound by
        # latency and launches
        dict(name="apply_tiny_f16", kind="apply", m=512, n=512, k=34, b=64, fmt="f16", round_x=False),
        # a server answering 16 queries at a time, all in 16 bits
        dict(name="apply_serve_f16o16", kind="apply", m=16384, n=16384, k=272, b=16, fmt="f16_o16", round_x=False),
        # an ordinary batch in binary32, of a matrix whose sides are odd
        dict(name="apply_mid_f32", kind="apply", m=12287, n=16381, k=272, b=250, fmt="f32", round_x=False),
        # queries arrive in binary64 and are rounded to the factors' format first
        dict(name="apply_round_bf16", kind="apply", m=16384, n=16384, k=272, b=4096, fmt="bf16", round_x=True),
        # the large batch in the paper's three precisions: the compensated
        # binary16 and binary32 factors and the binary64 baseline
        dict(name="apply_large_f16", kind="apply", m=16384, n=8192, k=144, b=8192, fmt="f16", round_x=False),
        dict(name="apply_large_f32", kind="apply", m=16384, n=8192, k=136, b=8192, fmt="f32", round_x=False),
        dict(name="apply_large_f64", kind="apply", m=16384, n=8192, k=128, b=8192, fmt="f64", round_x=False),
        # the paper's aggregate: ten matrices with sides up to 1138, one call
        dict(name="batched_f16", kind="batched", count=10, lo=400, hi=1138, k=41, b=8192, fmt="f16", sizes=4242),
        # a hyperspectral-shaped tensor, reconstructed from binary16 cores
        dict(name="tt_hsi_f16", kind="tt", dims="512,512,224", ranks="1,70,52,1", fmt="f16"),
        # a six-way tensor from binary32 cores
        dict(name="tt_six_f32", kind="tt", dims="16,16,16,16,16,16", ranks="1,16,26,26,26,16,1", fmt="f32"),
        # storing a matrix: round its binary64 factors, measure eta
        dict(name="store_matrix_f16", kind="store_matrix", m=16384, n=8192, k=144, fmt="f16"),
        # storing a tensor: round its cores, measure eta_TT, then check it
        # against the difference of the two dense binary64 reconstructions
        dict(name="store_tt_f16", kind="store_tt", dims="256,256,256", ranks="1,34,34,1", fmt="f16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_tt(rng, numel_max):
    if rng.random() < 0.6:
        dims = [_log_int(rng, 48, 512) for _ in range(3)]
        while math.prod(dims) > numel_max:
            i = dims.index(max(dims))
            dims[i] = max(32, int(dims[i] * 0.8))
        r = [_log_int(rng, 8, 70), _log_int(rng, 8, 52)]
    else:
        d = rng.randint(4, 6)
        top = {4: 60, 5: 27, 6: 16}[d]
        dims = [rng.randint(top // 2, top) for _ in range(d)]
        r = [rng.randint(8, 28)] * (d - 1)
    ranks = [1]
    for l in range(1, len(dims)):
        ranks.append(min(r[l - 1], math.prod(dims[:l]), math.prod(dims[l:])))
    ranks.append(1)
    return ",".join(map(str, dims)), ",".join(map(str, ranks))


def draw(rng):
    """One more case of the ranges above."""
    u = rng.random()
    fmt6 = ["f64", "f32", "f16", "f16_o16", "bf16", "f32tc"]
    if u < 0.55:
        fmt = rng.choice(["f64", "f64", "f32", "f32", "f16", "f16_o16", "bf16", "f32tc"])
        m, n = _log_int(rng, 512, 16384), _log_int(rng, 512, 16384)
        k = _log_int(rng, 24, 288)
        b = _log_int(rng, 1, 8192)
        # no binary64 case above the largest listed one's work
        while fmt == "f64" and (m + n) * k * b > 24576 * 128 * 8192:
            b = b * 3 // 4
        return dict(kind="apply", m=m, n=n, k=k, b=b, fmt=fmt, round_x=rng.random() < 0.25)
    if u < 0.65:
        return dict(kind="batched", count=rng.randint(4, 12), lo=400, hi=1138, k=rng.randint(32, 48),
                    b=_log_int(rng, 256, 8192), fmt=rng.choice(["f32", "f16", "f16_o16", "bf16"]),
                    sizes=rng.randint(1, 10 ** 6))
    if u < 0.85:
        dims, ranks = _draw_tt(rng, 512 * 512 * 224)
        return dict(kind="tt", dims=dims, ranks=ranks, fmt=rng.choice(fmt6))
    if u < 0.93:
        return dict(kind="store_matrix", m=_log_int(rng, 512, 16384), n=_log_int(rng, 512, 16384),
                    k=_log_int(rng, 24, 272), fmt=rng.choice(["f32", "f16", "bf16"]))
    dims, ranks = _draw_tt(rng, 256 ** 3)
    return dict(kind="store_tt", dims=dims, ranks=ranks, fmt=rng.choice(["f32", "f16", "bf16"]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _ints(text):
    return tuple(int(x) for x in text.split(","))


def _packed(rows, cols, dtype, gen, scale=None):
    """rows x cols seeded N(0, 1) values times `scale`, row pitch rounded up to
    16 elements (pad columns zero), drawn in binary64 and stored in `dtype`."""
    t = torch.zeros((rows, (cols + 15) // 16 * 16), dtype=dtype, device=DEV)
    step = max(1, (1 << 26) // max(cols, 1))
    for r in range(0, rows, step):
        v = torch.randn((min(step, rows - r), cols), generator=gen, dtype=torch.float64, device=DEV)
        if scale is not None:
            v *= scale
        t[r:r + step, :cols] = v.to(dtype)
    return t


def _matrix(m, n, k, dtype, gen):
    """Factors as a truncated SVD has them: nearly orthonormal columns of U and
    V, singular values j^-1.5."""
    U = _packed(m, k, dtype, gen, m ** -0.5)
    Vt = _packed(k, n, dtype, gen, n ** -0.5)
    s = torch.arange(1, k + 1, dtype=torch.float64, device=DEV) ** -1.5
    S = torch.zeros((1, (k + 15) // 16 * 16), dtype=dtype, device=DEV)
    S[0, :k] = s.to(dtype)
    return U, S, Vt


def _cores(dims, ranks, gen):
    """Cores of a TT in the left-orthogonal gauge (nearly orthonormal
    unfoldings, the last core scaled by 0.9^j), binary64."""
    out = []
    d = len(dims)
    for l in range(d):
        c = torch.randn((ranks[l], dims[l], ranks[l + 1]), generator=gen, dtype=torch.float64, device=DEV)
        if l < d - 1:
            c *= (ranks[l] * dims[l]) ** -0.5
        else:
            lam = 0.9 ** torch.arange(1, ranks[l] + 1, dtype=torch.float64, device=DEV)
            c *= dims[l] ** -0.5 * lam[:, None, None]
        out.append(c)
    return out


def _sizes(case):
    g = torch.Generator().manual_seed(case["sizes"])
    return torch.randint(case["lo"], case["hi"] + 1, (case["count"],), generator=g).tolist()


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    st = dict(case)
    kind, fmt = case["kind"], case["fmt"]
    dt, ot = lrc.storage_dtype(fmt), lrc.output_dtype(fmt)
    if kind == "apply":
        m, n, k, b = case["m"], case["n"], case["k"], case["b"]
        st["U"], st["S"], st["Vt"] = _matrix(m, n, k, dt, gen)
        if case["round_x"]:
            st["X64"] = _packed(b, n, torch.float64, gen)
            st["X"] = torch.empty(st["X64"].shape, dtype=dt, device=DEV)
        else:
            st["X"] = _packed(b, n, dt, gen)
        st["Y"] = torch.empty((b, m), dtype=ot, device=DEV)
    elif kind == "batched":
        k, b = case["k"], case["b"]
        st["sz"] = _sizes(case)
        fac = [_matrix(z, z, k, dt, gen) for z in st["sz"]]
        st["U"], st["S"], st["Vt"] = ([f[i] for f in fac] for i in range(3))
        st["X"] = [_packed(b, z, dt, gen) for z in st["sz"]]
        st["Y"] = [torch.empty((b, z), dtype=ot, device=DEV) for z in st["sz"]]
    elif kind == "tt":
        dims, ranks = _ints(case["dims"]), _ints(case["ranks"])
        st["d"], st["r"] = dims, ranks
        st["cores"] = [c.to(dt) for c in _cores(dims, ranks, gen)]
        st["out"] = torch.empty(math.prod(dims), dtype=ot, device=DEV)
    elif kind == "store_matrix":
        m, n, k = case["m"], case["n"], case["k"]
        st["f64"] = _matrix(m, n, k, torch.float64, gen)
        st["low"] = [torch.empty(t.shape, dtype=dt, device=DEV) for t in st["f64"]]
    else:
        dims, ranks = _ints(case["dims"]), _ints(case["ranks"])
        st["d"], st["r"] = dims, ranks
        st["f64"] = _cores(dims, ranks, gen)
        st["low"] = [torch.empty(c.shape, dtype=dt, device=DEV) for c in st["f64"]]
        st["wide"] = [torch.empty(c.shape, dtype=torch.float64, device=DEV) for c in st["f64"]]
        st["T"] = torch.empty(math.prod(dims), dtype=torch.float64, device=DEV)
        st["Th"] = torch.empty(math.prod(dims), dtype=torch.float64, device=DEV)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    kind, fmt = st["kind"], st["fmt"]
    if kind == "apply":
        m, n, k, b = st["m"], st["n"], st["k"], st["b"]
        if st["round_x"]:
            ld = st["X"].shape[1]
            lrc.lrc_round_factors(st["X64"], b, n, ld, st["X"], ld, fmt)
        lrc.lrc_apply(st["U"], st["S"], st["Vt"], st["X"], st["Y"], m, n, k, b, fmt)
        return [st["Y"]]
    if kind == "batched":
        c = st["count"]
        lrc.lrc_apply_batched(st["U"], st["S"], st["Vt"], st["X"], st["Y"], st["sz"], st["sz"], [st["k"]] * c,
                              [st["b"]] * c, fmt)
        return list(st["Y"])
    if kind == "tt":
        lrc.tt_reconstruct(st["cores"], st["d"], st["r"], fmt, st["out"])
        return [st["out"]]
    if kind == "store_matrix":
        m, n, k = st["m"], st["n"], st["k"]
        for src, dst, rows, cols in zip(st["f64"], st["low"], (m, 1, k), (k, k, n)):
            lrc.lrc_round_factors(src, rows, cols, src.shape[1], dst, dst.shape[1], fmt)
        eta, norm = lrc.lrc_lowrank_eta(*st["f64"], *st["low"], fmt, m, n, k)
        return [*st["low"], eta, norm]
    for src, dst in zip(st["f64"], st["low"]):
        rows, cols = src.shape[0], src.shape[1] * src.shape[2]
        lrc.lrc_round_factors(src, rows, cols, cols, dst, cols, fmt)
    eta, norm = lrc.lrc_tt_eta(st["f64"], st["low"], st["d"], st["r"], fmt)
    for src, dst in zip(st["low"], st["wide"]):
        rows, cols = src.shape[0], src.shape[1] * src.shape[2]
        lrc.lrc_widen_factors(src, fmt, rows, cols, cols, dst, cols)
    lrc.tt_reconstruct(st["f64"], st["d"], st["r"], "f64", st["T"])
    lrc.tt_reconstruct(st["wide"], st["d"], st["r"], "f64", st["Th"])
    diff, norm_dense = lrc.lrc_fro_diff(st["T"], "f64", st["Th"], "f64", st["T"].numel())
    return [*st["low"], eta, norm, st["T"], st["Th"], diff, norm_dense]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

_BYTES = {"f64": 8, "f32": 4, "f32tc": 4, "f16": 2, "f16_o16": 2, "bf16": 2}
_OUT = {"f64": 8, "f32": 4, "f32tc": 4, "f16": 4, "f16_o16": 2, "bf16": 2}


def _apply_work(m, n, k, b, fmt):
    e = _BYTES[fmt]
    return (m + n + 1) * k * e + b * n * e + b * m * _OUT[fmt], 2 * (m + n) * k * b + k * b


def _tt_flops(dims, ranks):
    """Multiply-adds (x 2) of the cheapest exact contraction that meets at one bond."""
    d = len(dims)
    best = None
    for c in range(1, d):
        f, p = 0, dims[0]
        for j in range(1, c):
            f += 2 * p * ranks[j] * dims[j] * ranks[j + 1]
            p *= dims[j]
        q = dims[d - 1]
        for j in range(d - 2, c - 1, -1):
            f += 2 * ranks[j] * dims[j] * ranks[j + 1] * q
            q *= dims[j]
        f += 2 * p * q * ranks[c]
        best = f if best is None else min(best, f)
    return best


def work(case):
    kind, fmt = case["kind"], case["fmt"]
    e = _BYTES[fmt]
    if kind == "apply":
        m, n, k, b = case["m"], case["n"], case["k"], case["b"]
        nbytes, flops = _apply_work(m, n, k, b, fmt)
        if case["round_x"]:
            nbytes += b * n * 8
        return {"bytes": nbytes, "flops": flops}
    if kind == "batched":
        w = [_apply_work(z, z, case["k"], case["b"], fmt) for z in _sizes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "store_matrix":
        m, n, k = case["m"], case["n"], case["k"]
        # binary64 factors read, stored factors written; the Gram matrices of
        # [dU, Uh] and [dV, Vh]
        return {"bytes": (m + n + 1) * k * (8 + e), "flops": 2 * (m + n) * k * (2 * k + 1)}
    dims, ranks = _ints(case["dims"]), _ints(case["ranks"])
    cores = sum(ranks[l] * dims[l] * ranks[l + 1] for l in range(len(dims)))
    numel = math.prod(dims)
    if kind == "tt":
        return {"bytes": cores * e + numel * _OUT[fmt], "flops": _tt_flops(dims, ranks)}
    # both dense tensors are results (written); their difference is read back
    return {"bytes": cores * (8 + e) + numel * 16, "flops": 2 * _tt_flops(dims, ranks) + 3 * numel}


def tolerance(case):
    """Relative 2-norm differences between two correct implementations: about
    four times the largest distance from `exact` measured over these ranges."""
    kind, fmt = case["kind"], case["fmt"]
    if kind in ("store_matrix", "store_tt"):
        # binary64 throughout; the difference of the two dense tensors loses
        # what they share, most where the stored cores are close to binary64
        return {"rel": 1e-11 if fmt == "f32" else 1e-13}
    if kind == "tt" and fmt == "f16":
        return {"rel": 4e-5}
    return {"rel": {"f64": 1.5e-14, "f32": 3e-6, "f32tc": 3e-6, "f16": 5e-6, "f16_o16": 1.2e-3, "bf16": 1e-2}[fmt]}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _rounded(x, dtype):
    """binary64 values rounded once to `dtype` (torch converts a double to 16
    bits through binary32; rounding to odd on the way makes that exact)."""
    f = x.float()
    if dtype == torch.float32 or dtype == torch.float64:
        return x.to(dtype)
    wide = f.double()
    bits = f.view(torch.int32) - (wide.abs() > x.abs()).int()
    return (bits | (wide != x).int()).view(torch.float32).to(dtype)


def _parts(x, dim, bits):
    """x as four terms, each a multiple of 2^-bits of the largest entry of what
    is left along `dim` (exact: all scales are powers of two)."""
    out = []
    for _ in range(4):
        e = torch.frexp(x.abs().amax(dim, keepdim=True))[1]
        t = torch.ldexp(torch.round(torch.ldexp(x, bits - e)), e - bits)
        out.append(t)
        x = x - t
    return out


def _mm(a, b):
    """a @ b as an unevaluated sum hi + lo of two binary64 matrices: the
    products of the parts are sums of integers below 2^53, so binary64 forms
    them without error."""
    bits = (52 - math.ceil(math.log2(max(2, a.shape[1])))) // 2
    pa, pb = _parts(a, 1, bits), _parts(b, 0, bits)
    hi = torch.zeros((a.shape[0], b.shape[1]), dtype=torch.float64, device=DEV)
    lo = torch.zeros_like(hi)
    for w in range(4):
        for i in range(w + 1):
            p = pa[i] @ pb[w - i]
            s = hi + p
            z = s - hi
            lo += (hi - (s - z)) + (p - z)
            hi = s
    s = hi + lo
    return s, lo - (s - hi)


def _mm2(a, lo, b):
    """(a + lo) @ b, lo small."""
    hi, rest = _mm(a, b)
    rest = rest + lo @ b
    s = hi + rest
    return s, rest - (s - hi)


def _exact_apply(U, S, Vt, X, m, n, k):
    """[(X V) diag(s)] U^T in binary64, in blocks of rows; where the operands
    are binary64 themselves, with sums carried in two of them."""
    V = Vt[:, :n].double().t()
    s = S[0, :k].double()
    Ut = U[:, :k].double().t()
    out = torch.empty((X.shape[0], m), dtype=torch.float64, device=DEV)
    step = 2048
    for r in range(0, X.shape[0], step):
        x = X[r:r + step, :n].double()
        if X.dtype == torch.float64:
            w, lo = _mm(x, V)
            # w s = p + q with q its rounding error (split by 27 bits)
            p = w * s
            wh, sh = 134217729.0 * w - (134217729.0 * w - w), 134217729.0 * s - (134217729.0 * s - s)
            wl, sl = w - wh, s - sh
            q = ((wh * sh - p) + wh * sl + wl * sh) + wl * sl
            out[r:r + step] = _mm2(p, q + lo * s, Ut)[0]
        else:
            out[r:r + step] = ((x @ V) * s) @ Ut
    return out


def _exact_tt(cores, wide=False):
    z = cores[0].double().reshape(cores[0].shape[1], -1)
    lo = torch.zeros_like(z)
    for c in cores[1:]:
        k = c.double().reshape(c.shape[0], -1)
        if wide:
            z, lo = (t.reshape(-1, c.shape[2]) for t in _mm2(z, lo, k))
        else:
            z = (z @ k).reshape(-1, c.shape[2])
    return z.reshape(-1)


def exact(case, seed):
    st = prepare(case, seed)
    kind, fmt = case["kind"], case["fmt"]
    dt = lrc.storage_dtype(fmt)
    if kind == "apply":
        X = _rounded(st["X64"], dt) if case["round_x"] else st["X"]
        return [_exact_apply(st["U"], st["S"], st["Vt"], X, case["m"], case["n"], case["k"])]
    if kind == "batched":
        return [_exact_apply(st["U"][p], st["S"][p], st["Vt"][p], st["X"][p], z, z, case["k"])
                for p, z in enumerate(st["sz"])]
    if kind == "tt":
        return [_exact_tt(st["cores"], fmt == "f64")]
    if kind == "store_matrix":
        n, k = case["n"], case["k"]
        U, S, Vt = st["f64"]
        Uh, Sh, Vh = (_rounded(t, dt).double() for t in st["f64"])
        # Gram factors of [dU, Uh] and [dV, Vh]: A - Ah = dU S V^T + Uh S dV^T + Uh dS Vh^T
        ru = torch.linalg.qr(torch.cat([(U - Uh)[:, :k], Uh[:, :k]], 1), mode="r")[1]
        rv = torch.linalg.qr(torch.cat([(Vt - Vh)[:, :n], Vh[:, :n]], 0).t(), mode="r")[1]
        du, uh, dv, vh = ru[:, :k], ru[:, k:], rv[:, :k], rv[:, k:]
        s, sh = S[0, :k], Sh[0, :k]
        v = dv + vh
        diff = (du * s) @ v.t() + (uh * s) @ dv.t() + (uh * (s - sh)) @ vh.t()
        norm = (((du + uh) * s) @ v.t()).norm()
        return [None, None, None, float(diff.norm()), float(norm)]
    low = [_rounded(c, dt) for c in st["f64"]]
    T, Th = _exact_tt(st["f64"], True), _exact_tt(low, True)
    eta, norm = float((T - Th).norm()), float(T.norm())
    return [*([None] * len(low)), eta, norm, T, Th, eta, norm]
