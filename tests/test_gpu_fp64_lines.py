"""Accuracy of long dense lines in the FP64 solver's fixed-point transforms."""
import math

import numpy as np
import pytest

from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc

pytestmark = pytest.mark.gpu


def _dct_solve_1d(g, d):
    """sum_k c_k(i) (sum_j c_k(j) g_j) / d_k in long double, the cosines from a table of 4 N angles."""
    N = g.size
    table = np.cos(np.arange(4 * N, dtype=np.longdouble) * (2 * np.arctan(np.longdouble(1)) / N))   # pi m / 2N
    i = np.arange(N, dtype=np.int64)
    u = np.zeros(N, dtype=np.longdouble)
    for k0 in range(0, N, 256):
        k = np.arange(k0, k0 + 256, dtype=np.int64)
        c = table[(k[:, None] * (2 * i[None, :] + 1)) % (4 * N)]
        x = (c * g[None, :]).sum(1) * np.where(k == 0, 1, 2) / N / d[k]
        u += (c * x[:, None]).sum(0)
    return u


@pytest.mark.parametrize("mean", [0.0, -1.0])
@pytest.mark.parametrize("N", [1024, 4096, 8192])
def test_dense_lines_are_as_accurate_as_fp64_ones(N, mean):
    """A field that varies along x alone: noise, and noise on a constant four
    times as large.  Two passes of log2 N butterfly levels and four more
    roundings (two factors of a pair, the normalisation, the result), each of up
    to 2^-53 and independent: 2^-53 sqrt(2 (log2 N + 4)) of the 2-norm."""
    import torch
    B.build()
    cc.load()
    g = mean + 0.25 * np.random.default_rng(N).standard_normal(N)
    c = (1.0, 0.25 / N**2, 0.0)
    k = np.arange(N, dtype=np.longdouble)
    s = 4 * np.longdouble(N) ** 2 * np.sin(k * (2 * np.arctan(np.longdouble(1)) / N)) ** 2
    want = _dct_solve_1d(g.astype(np.longdouble), np.longdouble(c[0]) + np.longdouble(c[1]) * s)
    solver = cc.SpectralSolver(N, 1.0, "neumann", "fp64")
    f = torch.from_numpy(g).cuda().expand(N, N).contiguous()
    u = solver.solve(c, f)
    solver.sync()
    got = u[N // 3].cpu().numpy().astype(np.longdouble)
    solver.close()
    e = float(np.sqrt(((got - want) ** 2).sum() / (want**2).sum()))
    print(N, mean, e)
    assert e <= 2.0**-53 * math.sqrt(2 * (math.log2(N) + 4))
