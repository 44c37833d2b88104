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


@pytest.mark.parametrize("N", [64, 256])
@pytest.mark.parametrize("scale", [1e3, 30.0, 1e-2, 1e-4, 1e-6, 1e-9, 1e-100])
def test_unit_of_the_concentration(N, scale, monkeypatch):
    """The same vesicle with the concentration in another unit."""
    w = I.workload("one_vesicle", N=N, dt=1e-7 / max(1.0, scale * scale))
    p = w.params.replace(psi_in=scale * w.params.psi_in, psi_out=scale * w.params.psi_out)
    _assert_same(*_both(monkeypatch, p, w.phi0, scale * w.psi0))


@pytest.mark.parametrize("N", [64, 256])
@pytest.mark.parametrize("amp", [1e-2, 1e-4, 1e-6])
def test_concentration_close_to_the_preferred_one(N, amp, monkeypatch):
    """psi within amp of psi_in = psi_out: f is gamma/2 (psi - psi_in)^2.  FP64
    rounds psi* by 2^-54, relative to the smallest |psi - psi_in| (0.05 amp) 2^-49 / amp;
    I_Z is twice as far off, its root as far as that."""
    w = I.workload("one_vesicle", N=N, dt=1e-7)
    p = w.params.replace(psi_in=0.65, psi_out=0.65)
    got, want = _both(monkeypatch, p, w.phi0, 0.65 + amp * (w.psi0 - 0.65))
    _assert_same(got, want, 1e-12 + 2.0**-49 / amp)


@pytest.mark.parametrize("ratio", [1e-1, 1e-2, 1e-4, 0.0])
def test_concentration_far_below_the_preferred_one(ratio, monkeypatch):
    """psi against psi_in and psi_out of order one, down to the FP64 stencil's
    part (means below 1/32 of them) and to psi = 0."""
    w = I.workload("one_vesicle", N=128, dt=1e-9)
    got, want = _both(monkeypatch, w.params, w.phi0, ratio * w.psi0)
    _assert_same(got, want)


@pytest.mark.parametrize("bg", [(1e-3, -2e-3), (2e4, 7e4), (5e9, 5e9)])
@pytest.mark.parametrize("gamma", [0.0, 1e2, 1e5])
def test_osmotic_constants(gamma, bg, monkeypatch):
    """beta_in, beta_out far below and far above gamma psi^2."""
    w = I.workload("one_vesicle", N=128, dt=1e-9)
    p = w.params.replace(gamma_in=gamma, gamma_out=2.0 * gamma, beta_in=bg[0], beta_out=bg[1])
    if gamma == 0.0:
        p = p.replace(beta_out=abs(bg[1]))
    _assert_same(*_both(monkeypatch, p, w.phi0, w.psi0))


@pytest.mark.parametrize("beta", [0.0, 1e-3, 0.3])
@pytest.mark.parametrize("amp", [1e-12, 1e-10, 1e-9, 1e-7, 1e-5, 1e-4, 1e-3])
@pytest.mark.parametrize("N", [64, 512])
def test_savs_of_a_state_without_an_interface(N, amp, beta, monkeypatch):
    """phi between 1 - 2.5 amp and 1 - 0.5 amp: the radicands are sums of terms of
    size amp^2 (I_V: about beta^2), so the SAVs show their accuracy.  FP64 rounds
    phi* and phi*^2 by 2^-54, relative to |phi*^2 - 1| >= amp 2^-53 / amp; four
    times that for the terms of a step."""
    p = I.growth_params(eps=8.0 / N, dt=1e-6, L=1.0, beta=beta)
    x = (np.arange(N) + 0.5) / N
    phi = 1.0 - amp * (1.5 + np.cos(np.pi * x)[None, :] * np.cos(2 * np.pi * x)[:, None])
    psi = 0.5 + 0.1 * np.cos(np.pi * x)[:, None] * np.ones(N)[None, :]
    got, want = _both(monkeypatch, p, phi, psi, 3)
    _assert_same(got, want, 1e-12 + 2.0**-51 / amp)


@pytest.mark.parametrize("beta", [0.0, 0.1, 0.3, 1.0])
def test_mean_of_phi_with_a_stiff_bending_term(beta, monkeypatch):
    """f0' holds beta phi_bar beside a bending term of coefficients ten million
    times larger; in the bulk it is the same in all cells.  Two steps of three
    roundings at |phi| = 1 (phi_bar, the increment, the sum) on either path:
    2e-15."""
    w = I.workload("one_vesicle", N=2048)
    got, want = _both(monkeypatch, w.params.replace(beta=beta, gamma_bend=1.0, dt=1e-4), w.phi0, w.psi0)
    assert abs((got[0] - want[0]).mean()) <= 2e-15
