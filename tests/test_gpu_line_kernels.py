"""Edges of the FP64 fixed-point kernels and the FP32 wide-line solver: scales
and non-finite values of a line, tiles outside the fixed-point stencil's range,
and coefficients outside the FP32 divisor's."""
import numpy as np
import pytest

from oracle import ccmsav_oracle as O
from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc
from paper_2601_10057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    return cc.load()


def _solve(f, coef, bc="neumann", precision="fp64", L=1.0):
    import torch
    s = cc.SpectralSolver(f.shape[0], L, bc, precision)
    t = torch.from_numpy(f).cuda().to(torch.float64 if precision == "fp64" else torch.float32).contiguous()
    u = s.solve(coef, t)
    s.sync()
    out = u.double().cpu().numpy()
    s.close()
    return out


# 64: the shortest fixed-point line, 256: several lanes' lines in a warp, 4096: a line on four warps
@pytest.mark.parametrize("N", [64, 256, 4096])
@pytest.mark.parametrize("k", [-700, 700])
def test_scaling_a_field_by_a_power_of_two_scales_the_solution_exactly(N, k):
    """A line's fixed-point scale is a power of two, so the arithmetic between
    the conversions does not depend on it: the bits agree."""
    f = np.random.default_rng(N).standard_normal((N, N))
    f[: N // 8] = 0.0                                    # zero lines
    f[:, 3] *= 1e-30                                     # values far below their line's largest
    coef = (1.5, 0.25 / N**2, 1e-3 / N**4)
    assert np.array_equal(_solve(np.ldexp(f, k), coef), np.ldexp(_solve(f, coef), k))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_does_not_come_back_finite(bad):
    f = np.ones((128, 128))
    f[17, 5] = bad
    assert not np.isfinite(_solve(f, (1.0, 1e-4, 0.0))).any()


def test_zero_field_solves_to_zero():
    assert not _solve(np.zeros((64, 64)), (2.0, 0.1, 0.0)).any()


# fractions of the grid that are too steep for the fixed-point range: none, one
# tile, about half the tiles, all of them
@pytest.mark.parametrize("N", [64, 512])
@pytest.mark.parametrize("part", [0.0, 0.01, 0.5, 1.0])
def test_steep_tiles_match_the_block_path(N, part, monkeypatch):
    """Two steps from a state whose first rows carry cell-to-cell jumps of phi
    above 1/4 (those tiles are evaluated in FP64), against the FP64 stencil and
    block transforms on the whole grid.  A few hundred roundings of 1e-16 along
    two steps: 1e-12 of the largest value."""
    w = I.workload("one_vesicle", N=N, dt=1e-7)
    phi = w.phi0.copy()
    rows = int(round(part * N))
    phi[:rows] += 0.3 * np.random.default_rng(1).uniform(-1.0, 1.0, (rows, N))
    out = []
    for block in ("0", "1"):
        monkeypatch.setenv("CCMSAV_FORCE_BLOCK_FFT", block)       # read when the handle is created
        sim = cc.Simulation(w.params, N, precision="fp64")
        sim.set_state(phi, w.psi0)
        sim.step(2)
        out.append(sim.state())
        sim.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


@pytest.mark.parametrize("coef", [(-3.0, 1.0, 0.0), (1e30, 1e26, 1e20), (2.0, 0.1, 1e-6)])
def test_fp32_coefficients_in_and_outside_the_divisors_range(coef):
    """Dirichlet, N = 64: a negative c0 and divisors above the FP32 pairs' range
    (both solved by the block kernels) and an ordinary one; 2e-5 as in the
    solver's other FP32 parity tests."""
    f = np.random.default_rng(3).standard_normal((64, 64))
    want = O.spectral_solve_bc(f, coef, 1.0 / 64, "dirichlet")
    got = _solve(f, coef, "dirichlet", "fp32")
    assert np.abs(got - want).max() <= 2e-5 * np.abs(want).max()


@pytest.mark.parametrize("N", [32, 64, 1024])
def test_periodic_fp32_against_fp64(N):
    """Half-spectrum transforms (from N = 64) against the FP64 solver."""
    f = np.random.default_rng(N).standard_normal((N, N))
    coef = (1.0, 4.0 / N**2, 1.0 / N**4)
    want = _solve(f.astype(np.float32).astype(np.float64), coef, "periodic")
    got = _solve(f, coef, "periodic", "fp32")
    assert np.abs(got - want).max() <= 2e-5 * np.abs(want).max()


@pytest.mark.parametrize("amp", [1e-12, 1e-9, 1e-4])
def test_state_without_an_interface(amp, monkeypatch):
    """phi within amp of 1 everywhere: the SAV radicands are sums of terms of
    size amp^2, far below the fixed-point fields' last bit for the smaller
    ones.  The run goes on as on the block path, within 1e-12 of the largest value."""
    N = 128
    p = I.growth_params(eps=8.0 / N, dt=1e-6, L=1.0)
    x = (np.arange(N) + 0.5) / N
    phi = 1.0 - amp * (1.5 + np.cos(np.pi * x)[None, :] * np.cos(2 * np.pi * x)[:, None])
    psi = 0.5 + 0.1 * np.cos(np.pi * x)[:, None] * np.ones(N)[None, :]
    out = []
    for block in ("0", "1"):
        monkeypatch.setenv("CCMSAV_FORCE_BLOCK_FFT", block)
        sim = cc.Simulation(p, N, precision="fp64")
        sim.set_state(phi, psi)
        sim.step(3)
        out.append(sim.state())
        sim.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


@pytest.mark.parametrize("wl,N", [("ellipse_shrink", 64), ("three_vesicles", 1024), ("three_vesicles", 4096)])
def test_classical_fp32_preconditioner_lines(wl, N):
    """FP32 conjugate gradients to 1e-6, preconditioned on the wide lines (the
    shortest, a middle and the clustered ones), against FP64 after 2 steps: 2e-5, the CG
    tolerance and the FP32 fields' rounding over the steps."""
    w = I.workload(wl, N=N, dt=1e-6)
    out = []
    for prec, tol in (("fp64", 1e-10), ("fp32", 1e-6)):
        sim = cc.Simulation(w.params, N, precision=prec, classical=True)
        sim.set_pcg(tol, 400)
        sim.set_state(w.phi0, w.psi0)
        sim.step(2)
        out.append(sim.state())
        assert 1 <= sim.pcg_stats()[0] < 400
        sim.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 2e-5 * np.abs(a).max()
