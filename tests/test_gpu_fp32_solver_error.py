"""Rounding error of the FP32 solver's wide lines against that of the general
block kernels on the same inputs."""
import math

import numpy as np
import pytest

from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc
from paper_2601_10057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["neumann", "dirichlet", "periodic"])
def test_error_is_no_larger_than_the_general_kernels(bc):
    """Coefficients times 2^90 lie outside the wide lines' range and take the
    general kernels; the solution is 2^-90 times as large, exactly.  Geometric
    mean of the error ratio over sizes, smoothing widths and fields (an interface
    field with noise): at most 1."""
    import torch
    B.build()
    cc.load()
    logs, big = [], 2.0**90
    for N in (256, 512, 1024, 2048, 4096):
        s, d = cc.SpectralSolver(N, 1.0, bc, "fp32"), cc.SpectralSolver(N, 1.0, bc, "fp64")
        phi = torch.from_numpy(I.workload("one_vesicle", N=N).phi0).cuda()
        for seed in range(3):
            g = torch.Generator(device="cpu").manual_seed(seed)
            f = (phi + 0.25 * torch.randn(N, N, generator=g).cuda().double()).float().contiguous()
            for cells in (0.5, 3.0, 40.0):
                w = (cells / N) ** 2
                c = (1.0, w, 0.1 * w * w)
                want = d.solve(c, f.double().contiguous())
                d.sync()
                wide = s.solve(c, f)
                s.sync()
                general = s.solve(tuple(big * x for x in c), f)
                s.sync()
                e = [float((u - want).norm() / want.norm()) for u in (wide.double(), general.double() * big)]
                logs.append(math.log(e[0] / e[1]))
                print(bc, N, cells, seed, e)
        s.close()
        d.close()
    mean = math.exp(sum(logs) / len(logs))
    print(bc, "mean ratio", mean, "largest", math.exp(max(logs)))
    assert mean <= 1.0
