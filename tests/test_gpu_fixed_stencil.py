"""The FP64 stencil in 64-bit fixed point against the FP64 stencil (block path)
at the edges of its number formats: large normalised sums, concentrations and
osmotic terms of any size, states without an interface."""
import math

import numpy as np
import pytest

from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc
from paper_2601_10057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    return cc.load()


def _both(monkeypatch, p, phi, psi, steps=2):
    """(phi, psi, SAVs V U W Z) after ``steps`` steps on the fixed-point and on the block path."""
    out = []
    for block in ("0", "1"):
        monkeypatch.setenv("CCMSAV_FORCE_BLOCK_FFT", block)       # read when the handle is created
        sim = cc.Simulation(p, phi.shape[0], precision="fp64")
        sim.set_state(phi, psi)
        sim.step(steps)
        out.append(sim.state() + (np.array(sim.aux()[:4]),))
        sim.close()
    return out


def _assert_same(got, want, savs=1e-12):
    """Fields within 1e-12 of the largest value (some hundred roundings of
    1e-16 along two steps), each SAV within ``savs`` of itself."""
    for a, b in zip(got[:2], want[:2]):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
    assert (np.abs(got[2] - want[2]) <= savs * np.abs(want[2]))[[0, 2, 3]].all(), (got[2], want[2])


def _half_zero(N, L):
    """0 in one half, rising to 1 over an interface of 16 cells."""
    x = (np.arange(N) + 0.5) * (L / N)
    return 0.5 * (1.0 + np.tanh((x - 0.6 * L) / (math.sqrt(2.0) * 8.0 * L / N)))[None, :] * np.ones((N, 1))


# the tiles of N = 2048 are the largest (a warp adds up to 288 cells)
@pytest.mark.parametrize("N", [256, 512, 2048])
@pytest.mark.parametrize("case", ["psi_out", "psi_negative", "gamma_ratio", "beta"])
def test_sums_of_large_terms(N, case, monkeypatch):
    """Normalised terms of I_Z and I_V as large as the parameters allow, over
    whole tiles: psi far from psi_out (4.8 a cell at psi_out = 5 where psi = 0),
    negative concentrations, osmotic constants above the quadratic terms, and
    (phi^2 - 1 - beta)^2 = 4 where phi = 0 and beta = 1."""
    w = I.workload("one_vesicle", N=N, dt=1e-8)
    p, phi, psi = w.params, w.phi0, w.psi0
    if case == "psi_out":
        p, psi = p.replace(psi_out=5.0), psi - 0.8
    elif case == "psi_negative":
        psi = psi - 2.5
    elif case == "gamma_ratio":
        p, psi = p.replace(gamma_in=1e5, gamma_out=1e2, beta_in=3e4, beta_out=5e5), psi + 1.5
    else:
        p, phi = p.replace(beta=1.0), _half_zero(N, p.L)
    _assert_same(*_both(monkeypatch, p, phi, psi))
