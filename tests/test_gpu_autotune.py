"""Candidates of the autotuner, counted by the launches of the steps it times."""
import pytest

from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc
from paper_2601_10057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# three carveouts and the block transforms; at N = 8192 the kernels take no carveout
@pytest.mark.parametrize("N,candidates", [(128, 4), (8192, 2)])
def test_no_schedule_is_timed_twice(N, candidates):
    """Three warm-up and three timed steps of six launches a candidate."""
    B.build()
    cc.load()
    w = I.workload("one_vesicle", N=N, dt=1e-6)
    sim = cc.Simulation(w.params, N, precision="fp32")
    sim.set_state(w.phi0, w.psi0)
    sim.step(1)
    n = sim.launches()
    sim.autotune(3)
    assert sim.launches() - n == candidates * 6 * 6
    sim.close()
