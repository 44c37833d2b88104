"""Fields that start one value behind a 16-byte boundary: periodic solves take
them, the Neumann and Dirichlet ones refuse them."""
import numpy as np
import pytest

from oracle import ccmsav_oracle as O
from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc

pytestmark = pytest.mark.gpu
COEF = (1.5, 1e-3, 1e-8)


def _shifted(a, dtype):
    import torch
    t = torch.zeros(a.size + 1, dtype=dtype, device="cuda")[1:].view(a.shape)
    assert t.data_ptr() % 16 != 0
    return t.copy_(torch.from_numpy(a))


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    return cc.load()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [32, 64, 512])
def test_periodic_fields_at_any_address(N, precision):
    """Input, output or both shifted; the bounds of the solver's parity tests."""
    import torch
    dtype = torch.float64 if precision == "fp64" else torch.float32
    f = np.random.default_rng(N).standard_normal((N, N))
    want = O.spectral_solve_bc(f, COEF, 1.0 / N, "periodic")
    s = cc.SpectralSolver(N, 1.0, "periodic", precision)
    plain = torch.from_numpy(f).cuda().to(dtype)
    for src, dst in ((_shifted(f, dtype), torch.empty_like(plain)), (plain, _shifted(0 * f, dtype)),
                     (_shifted(f, dtype), _shifted(0 * f, dtype))):
        u = s.solve(COEF, src, out=dst)
        s.sync()
        assert np.abs(u.double().cpu().numpy() - want).max() <= (1e-12 if precision == "fp64" else 2e-5) * np.abs(want).max()
    s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bc", ["neumann", "dirichlet"])
def test_other_boundaries_refuse_unaligned_fields(bc, precision):
    import torch
    N, dtype = 64, torch.float64 if precision == "fp64" else torch.float32
    s = cc.SpectralSolver(N, 1.0, bc, precision)
    f = np.ones((N, N))
    ok = torch.ones(N, N, dtype=dtype, device="cuda")
    for src, dst in ((_shifted(f, dtype), ok), (ok, _shifted(f, dtype))):
        with pytest.raises(cc.CCMSAVError):
            s.solve(COEF, src, out=dst)
    with pytest.raises(cc.CCMSAVError):
        s.smooth(_shifted(f, dtype), 0.1)
    s.close()
