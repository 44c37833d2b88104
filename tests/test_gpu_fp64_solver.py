"""The FP64 Neumann solve keeps the division of each mode correctly rounded."""
import numpy as np
import pytest

from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc

pytestmark = pytest.mark.gpu


def test_division_of_a_mode_is_correctly_rounded():
    """A constant field a has one mode, 64 a at N = 64, whose transforms only
    multiply by powers of two: u is a / c0 rounded once."""
    import torch
    B.build()
    cc.load()
    N = 64
    s = cc.SpectralSolver(N, 1.0, "neumann", "fp64")
    f, u = torch.empty(N, N, dtype=torch.float64, device="cuda"), torch.empty(N, N, dtype=torch.float64, device="cuda")
    for a, c0 in np.random.default_rng(N).uniform(1.0, 2.0, (500, 2)):
        s.solve((float(c0), 1e-3, 1e-6), f.fill_(float(a)), out=u)
        s.sync()
        assert bool((u == float(a) / float(c0)).all()), (a, c0)
    s.close()
