"""Rounding to the 16-bit formats by integer operations: bit-exact against the
oracle at every midpoint and neighbour of the format, at its limits, and for a
source that lies in one run, one that starts off a 32-byte boundary, and one
whose rows are not whole groups."""
import numpy as np
import pytest
import torch

import oracle
from parity import bits

pytestmark = pytest.mark.gpu


def _values(fmt):
    top = 0x7C00 if fmt == "f16" else 0x7F80
    pos = oracle.decode(np.arange(0, top, dtype=np.uint16), fmt)
    mid = (pos[:-1] + pos[1:]) / 2.0
    big = pos[-1] + (pos[-1] - pos[-2]) / 2.0           # rounds to infinity
    x = np.concatenate([pos, mid, np.nextafter(mid, np.inf), np.nextafter(mid, 0.0),
                        [big, np.nextafter(big, 0.0), 2 * big, 1e300, 5e-324, 2.2e-308, np.inf, 0.0]])
    return np.concatenate([x, -x])


@pytest.mark.parametrize("fmt", ["f16", "bf16"])
@pytest.mark.parametrize("cols,first", [(8, 0), (4096, 0), (64, 2), (64, 4), (61, 0), (7, 0)])
def test_every_midpoint(lrc, cuda, fmt, cols, first):
    x = _values(fmt)
    rows = -(-x.size // cols)
    flat = np.zeros(first + rows * cols)
    flat[first:first + x.size] = x
    src = torch.from_numpy(flat).to(cuda)[first:].view(rows, cols)
    got = bits(lrc.round_matrix(src, fmt, ld=cols), fmt)
    torch.cuda.synchronize()
    want = oracle.round_bits(flat[first:], fmt).reshape(rows, cols)
    assert np.array_equal(got, want)
