"""Index-checked runs (libccmsav_bounds.so) of the line kernels that
tests/test_gpu_bounds.py does not reach: the solver at every line length, the
FP64 step of the large grids and the FP32 classical preconditioner, in a child
process; no access may leave its array."""
import json
import os
import subprocess
import sys

import pytest

from paper_2601_10057_gb300 import build as B
from paper_2601_10057_gb300 import ccmsav as cc

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
import torch
sys.path.insert(0, sys.argv[1])
from paper_2601_10057_gb300 import ccmsav as cc
from paper_2601_10057_gb300 import inputs as I
cc.load(cc.LIB_BOUNDS_PATH)
out = []
for lg in range(6, 14):
    N = 1 << lg
    for bc in ("neumann", "dirichlet", "periodic"):
        for prec, dtype in (("fp64", torch.float64), ("fp32", torch.float32)):
            s = cc.SpectralSolver(N, 1.0, bc, prec)
            f = torch.ones(N, N, dtype=dtype, device="cuda")
            u = s.solve((2.0, 1e-4 / N, 1e-8 / N**2), f)
            s.sync()
            line = bc != "periodic" or (prec == "fp32" and N <= 4096)
            err = float((u - 0.5).abs().max()) if bc != "dirichlet" else 0.0
            out.append({"case": f"solve {N} {bc} {prec}", "flag": cc.ccmsav_solver_bounds_flag(s.h) if line else 0, "err": err})
            s.close()
for N in (512, 2048, 4096, 8192):
    w = I.workload("one_vesicle", N=N, dt=1e-7)
    for prec, classical in (("fp64", False), ("fp32", True)):
        sim = cc.Simulation(w.params, N, precision=prec, classical=classical)
        if classical:
            sim.set_pcg(1e-5, 50)
        sim.set_state(w.phi0, w.psi0)
        sim.step(3)
        sim.sync()
        out.append({"case": f"step {N} {prec}", "flag": cc.ccmsav_bounds_flag(sim.h), "err": 0.0})
        sim.close()
print(json.dumps(out))
"""


def test_line_kernels_stay_in_their_arrays():
    """A constant field's solve (one mode, within FP32's rounding of the
    transforms) and steps at the sizes whose kernels differ."""
    B.build(bounds=True)
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert all(c["flag"] == 0 for c in res), [c for c in res if c["flag"]]
    assert all(c["err"] <= 2e-5 for c in res), [c for c in res if c["err"] > 2e-5]


def test_the_flag_needs_a_checked_build():
    B.build()
    cc.load()
    s = cc.SpectralSolver(64, 1.0, "neumann", "fp32")
    assert cc.ccmsav_solver_bounds_flag(s.h) == -1
    s.close()
