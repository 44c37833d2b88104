"""set_state from host and from device memory."""
import numpy as np
import pytest

from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc
from paper_2601_10057_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [64, 512])
def test_host_and_device_fields_give_the_same_state(N):
    """FP32: the same SAVs and arc length (one kernel sums them either way) and
    the conserved mean to FP64's rounding of the two orders of summation."""
    import torch
    B.build()
    cc.load()
    w = I.workload("one_vesicle", N=N, dt=1e-6)
    phi, psi = (torch.from_numpy(f).cuda().float().contiguous() for f in (w.phi0, w.psi0))
    aux = []
    for device in (False, True):
        sim = cc.Simulation(w.params, N, precision="fp32")
        if device:
            assert cc.ccmsav_set_state_device(sim.h, 0, phi.data_ptr(), psi.data_ptr()) == cc.CCMSAV_OK
        else:
            sim.set_state(phi.double().cpu().numpy(), psi.double().cpu().numpy())
        aux.append(np.array(sim.aux()))
        sim.close()
    assert np.array_equal(aux[0][:9], aux[1][:9])
    assert abs(aux[0][11] - aux[1][11]) <= 1e-13 * abs(aux[1][11])


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("field", [0, 1])
def test_non_finite_device_fields_are_refused(field, bad):
    import torch
    B.build()
    cc.load()
    w = I.workload("one_vesicle", N=64, dt=1e-6)
    f = [torch.from_numpy(x).cuda().float().contiguous() for x in (w.phi0, w.psi0)]
    f[field][5, 7] = bad
    sim = cc.Simulation(w.params, 64, precision="fp32")
    assert cc.ccmsav_set_state_device(sim.h, 0, f[0].data_ptr(), f[1].data_ptr()) == cc.CCMSAV_ENONFINITE
    sim.close()
