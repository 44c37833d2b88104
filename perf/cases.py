"""Workloads of the CC-MSAV time stepper, the spectral solver and the smoother
as a user's program runs them, each through the public entry points.

A *step* case is one simulation run: the initial state is handed over in
device memory, ``steps`` time steps are queued and the final fields are
fetched into page-locked host buffers.  A *batch* case does the same for a
handle of many simulations, a *solve* case is one elliptic solve of a device
field and a *smooth* case the initial-condition smoother.

The fields of an FP32 simulation come back from ``ccmsav_get_state`` widened
to FP64; the program keeps them in the precision they were computed in.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2601_10057_gb300 import ccmsav
from paper_2601_10057_gb300 import inputs

SQ2 = math.sqrt(2.0)
L = 2 * math.pi
SIZES = (128, 256, 512)            # grid sizes of a batch's simulations


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _step(name, N, precision, steps, vesicles, dt=1e-5, scheme="cc", energy=False, column="growth"):
    c = {"kind": "step", "N": N, "precision": precision, "steps": steps, "vesicles": vesicles, "dt": dt,
         "scheme": scheme, "energy": energy, "column": column}
    return dict(c, name=name) if name else c


def _batch(name, sims, steps):
    c = {"kind": "batch", "sims": sims, "precision": "fp32", "steps": steps, "dt": 1e-5, "column": "shrinkage"}
    return dict(c, name=name) if name else c


def _solve(name, N, precision, bc, cells=3.0):
    c = {"kind": "solve", "N": N, "precision": precision, "bc": bc, "cells": cells}
    return dict(c, name=name) if name else c


def _smooth(name, N, precision, shape, bc="neumann", steps=10):
    c = {"kind": "smooth", "N": N, "precision": precision, "shape": shape, "bc": bc, "steps": steps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # one vesicle on a coarse grid, the quick look and parameter scan: latency and launches
        _step("step_fp64_n64", 64, "fp64", 200, 1, dt=1e-4),
        # a single shrinking or growing vesicle with the energy balance tracked, FP64 (the default precision)
        _step("step_fp64_n512_energy", 512, "fp64", 50, 1, energy=True),
        # the throughput workload's grid in the default precision
        _step("step_fp64_n2048", 2048, "fp64", 6, 3),
        # shrinking vesicles on a mid-size grid in FP32, where the kernels no longer fill the chip
        _step("step_fp32_n512", 512, "fp32", 300, 16, column="shrinkage"),
        # the throughput workload: three vesicles, FP32
        _step("step_fp32_n2048", 2048, "fp32", 200, 3),
        # the largest grid a handle takes
        _step("step_fp32_n8192", 8192, "fp32", 20, 16, dt=5e-6),
        # 64 simulations of mixed sizes in one handle: a parameter study
        _batch("batch_fp32_64", 64, 60),
        # the paper's baseline scheme (conjugate gradients in each step)
        _step("classical_fp64_n1024", 1024, "fp64", 3, 3, scheme="classical"),
        # one small elliptic solve: latency
        _solve("solve_dirichlet_fp64_n256", 256, "fp64", "dirichlet"),
        # a periodic solve between FP32 fields
        _solve("solve_periodic_fp32_n1024", 1024, "fp32", "periodic"),
        # a large Neumann solve in FP32
        _solve("solve_neumann_fp32_n4096", 4096, "fp32", "neumann"),
        # smoothing a sharp shape into an initial condition, at the robustness runs' size
        _smooth("smooth_fp64_n2048", 2048, "fp64", "star"),
    ]


def draw(rng):
    u = rng.random()
    if u < 0.55:
        precision = rng.choice(["fp64", "fp32"])
        scheme = rng.choice(["cc", "cc", "cc", "cc", "bdf1", "classical"])
        energy = precision == "fp64" and scheme == "cc" and rng.random() < 0.4
        top = 13 if precision == "fp32" else 12
        N = 1 << rng.randint(6, top if scheme != "classical" else 10)
        # points times steps, bounded well below the largest listed case's time
        cap = (1.2e9 if precision == "fp32" else 3.0e7) / (8 if scheme == "classical" else 1)
        most = max(2, min(300 if scheme != "classical" else 6, int(cap / (N * N))))
        steps = max(2, min(most, int(round(math.exp(rng.uniform(math.log(2), math.log(most + 1)))))))
        return _step(None, N, precision, steps, rng.choice([1, 3]) if precision == "fp64" else _many(N),
                     dt=5e-6 if N > 4096 else 1e-5, scheme=scheme, energy=energy,
                     column="shrinkage" if precision == "fp32" and N <= 512 else "growth")
    if u < 0.65:
        return _batch(None, rng.randint(3, 63), rng.randint(20, 70))
    if u < 0.9:
        return _solve(None, 1 << rng.randint(5, 12), rng.choice(["fp64", "fp32"]),
                      rng.choice(["neumann", "dirichlet", "periodic"]), round(rng.uniform(0.5, 40.0), 2))
    return _smooth(None, 1 << rng.randint(6, 12), rng.choice(["fp64", "fp64", "fp32"]),
                   rng.choice(list(inputs.SHARP_SHAPES)), steps=rng.randint(1, 10))


# ---------------------------------------------------------------- inputs

def _dtype(precision):
    return torch.float64 if precision == "fp64" else torch.float32


def _eps(N):
    """Four cells up to N = 2048, that physical width on larger grids."""
    return 4.0 * L / min(N, 2048)


def _many(N):
    """Vesicles of an FP32 simulation: close enough together (in interface widths) that
    no region between them is exactly -1.  Such a region is an unstable state of the
    model, from which rounding errors grow at first."""
    return 4 if N <= 64 else 9 if N <= 256 else 16


def _fields(N, count, seed, column="growth"):
    """phi and psi (FP64) of ``count`` perturbed circles on a jittered square
    lattice: growing and shrinking vesicles by turns, or shrinking ones only."""
    rng = np.random.Generator(np.random.PCG64(seed))
    dev, eps = _dev(), _eps(N)
    side = int(math.ceil(math.sqrt(count)))
    cell = L / side
    x = (torch.arange(N, dtype=torch.float64, device=dev) + 0.5) * (L / N)
    phi = torch.full((N, N), -1.0, dtype=torch.float64, device=dev)
    psi = torch.full((N, N), 0.8, dtype=torch.float64, device=dev)
    for k in range(count):
        R = cell * rng.uniform(0.18, 0.3)
        jit = max(0.0, cell / 2 - R * 1.15 - 4 * eps)
        jx, jy = rng.uniform(-1.0, 1.0, 2) * jit
        amps, phases = rng.uniform(0.0, 0.03, 5), rng.uniform(0.0, 2 * math.pi, 5)
        dx = x[None, :] - ((k % side + 0.5) * cell + jx)
        dy = x[:, None] - ((k // side + 0.5) * cell + jy)
        th, rad = torch.atan2(dy.expand(N, N), dx.expand(N, N)), 1.0
        for m, (a, p) in enumerate(zip(amps, phases), start=2):
            rad = rad + a * torch.cos(m * th + p)
        pk = torch.tanh((R * rad - torch.sqrt(dx * dx + dy * dy)) / (SQ2 * eps))
        inside = 0.1 if k % 2 == 0 and column == "growth" else 0.6
        phi = torch.maximum(phi, pk)
        psi = psi + (inside - 0.8) * (1.0 + pk) / 2.0
    return phi, psi


def _params(N, case):
    make = inputs.growth_params if case["column"] == "growth" else inputs.shrinkage_params
    return make(eps=_eps(N), dt=case["dt"], L=L)


def _batch_members(case, seed):
    """(N, field seed) of each simulation of a batch."""
    rng = np.random.Generator(np.random.PCG64(977 + case["sims"]))     # the sizes belong to the case
    return [(int(rng.choice(SIZES)), 10007 * seed + k) for k in range(case["sims"])]


def _solve_coef(case):
    """c0 - c1 Lap + c2 Lap^2 with both scales ``cells`` grid cells wide."""
    w = (case["cells"] / case["N"]) ** 2
    return [1.0, w, 0.1 * w * w]


def _solve_rhs(case, seed):
    """An interface field with noise on top."""
    N = case["N"]
    g = torch.Generator(device="cpu").manual_seed(seed)
    noise = torch.randn(N, N, generator=g, dtype=torch.float32).to(_dev())
    phi, _ = _fields(N, 3, seed)
    return (phi + 0.25 * noise.double()).to(_dtype(case["precision"])).contiguous()


def _smooth_input(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    phi = inputs.sharp_shape(case["shape"], case["N"], L=1.0, R=float(rng.uniform(0.15, 0.35)))
    return torch.from_numpy(phi).to(_dev()).to(_dtype(case["precision"])).contiguous()


def _smooth_args(case):
    return {"eps": 0.01 if case["N"] >= 512 else 5.12 / case["N"], "mobility": 0.01, "dt": 1e-6}


def _result_buffers(N, precision):
    """Page-locked FP64 buffers for get_state, and the FP32 arrays the program keeps."""
    out = [torch.empty(N, N, dtype=torch.float64, pin_memory=True) for _ in range(2)]
    keep = out if precision == "fp64" else [torch.zeros(N, N, dtype=torch.float32) for _ in range(2)]
    return out, keep


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        N, precision, scheme = case["N"], case["precision"], case["scheme"]
        sim = ccmsav.Simulation(_params(N, case), N, precision=precision, track_energy=case["energy"],
                                bdf1_always=scheme == "bdf1", classical=scheme == "classical")
        phi, psi = [f.to(_dtype(precision)).contiguous() for f in _fields(N, case["vesicles"], seed, case["column"])]
        out, keep = _result_buffers(N, precision)
        return {"case": case, "sim": sim, "members": [(phi, psi, out, keep)]}
    if kind == "batch":
        members = _batch_members(case, seed)
        sim = ccmsav.Simulation(None, [N for N, _ in members], precision=case["precision"],
                                per_sim=[_params(N, case) for N, _ in members])
        got = []
        for N, s in members:
            phi, psi = [f.to(_dtype(case["precision"])).contiguous() for f in _fields(N, _many(N), s, case["column"])]
            got.append((phi, psi) + _result_buffers(N, case["precision"]))
        return {"case": case, "sim": sim, "members": got}
    bc, N = case["bc"], case["N"]
    solver = ccmsav.SpectralSolver(N, 1.0, bc=bc, precision=case["precision"])
    f = _solve_rhs(case, seed) if kind == "solve" else _smooth_input(case, seed)
    return {"case": case, "solver": solver, "f": f, "u": torch.empty_like(f)}


# ---------------------------------------------------------------- one pass

_DP = ctypes.POINTER(ctypes.c_double)


def _check(status, where):
    if status != ccmsav.CCMSAV_OK:
        raise ccmsav.CCMSAVError(status, where)


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        state["solver"].solve(_solve_coef(case), state["f"], out=state["u"])
        state["solver"].sync()
        return state["u"]
    if case["kind"] == "smooth":
        state["u"].copy_(state["f"])
        state["solver"].smooth(state["u"], nsteps=case["steps"], **_smooth_args(case))
        state["solver"].sync()
        return state["u"]
    sim, lib = state["sim"], ccmsav.load()
    for k, (phi, psi, _, _) in enumerate(state["members"]):
        _check(ccmsav.ccmsav_set_state_device(sim.h, k, phi.data_ptr(), psi.data_ptr()), "ccmsav_set_state_device")
    sim.step(case["steps"])
    for k, (_, _, out, keep) in enumerate(state["members"]):
        _check(lib.ccmsav_get_state(sim.h, k, *(ctypes.cast(t.data_ptr(), _DP) for t in out)), "ccmsav_get_state")
        if keep is not out:
            for dst, src in zip(keep, out):
                dst.copy_(src)
    if case["kind"] == "batch":
        return {f: torch.cat([m[3][i].reshape(-1) for m in state["members"]]) for i, f in enumerate(("phi", "psi"))}
    phi, psi = state["members"][0][3]
    res = {"phi": phi, "psi": psi}
    if case["energy"]:
        res["energy"] = sim.energy()
    return res


def work(case):
    """One pass: per step 40 field passes (stencil 4 in, 8 fields through a forward
    and 2 through an inverse 2D transform, the Gram sums and the recovery between);
    per solve the field read and written."""
    size = 8 if case["precision"] == "fp64" else 4
    if case["kind"] in ("step", "batch"):
        sizes = [case["N"]] if case["kind"] == "step" else [N for N, _ in _batch_members(case, 0)]
        pts = sum(N * N for N in sizes)
        per_pt = 50 * math.log2(max(sizes)) + 320
        if case["kind"] == "step" and case["scheme"] == "classical":    # ten or more iterations on two systems
            return {"bytes": pts * size * case["steps"] * (40 + 200), "flops": pts * case["steps"] * (per_pt + 2000)}
        return {"bytes": pts * size * 40 * case["steps"], "flops": pts * case["steps"] * per_pt}
    pts = case["N"] ** 2
    n = case["steps"] if case["kind"] == "smooth" else 1
    return {"bytes": 2 * pts * size * n, "flops": pts * n * (10 * math.log2(case["N"]) + 20)}


# ---------------------------------------------------------------- 64-bit reference

def _dct(x, dim):
    """Orthonormal DCT-II along dim through one complex FFT of the even / odd reordered line."""
    x = x.transpose(dim, -1)
    N = x.shape[-1]
    v = torch.cat([x[..., ::2], x[..., 1::2].flip(-1)], -1)
    k = torch.arange(N, dtype=torch.float64, device=x.device)
    X = (torch.fft.fft(v) * torch.polar(torch.ones_like(k), -math.pi * k / (2 * N))).real * math.sqrt(2.0 / N)
    X[..., 0] /= SQ2
    return X.transpose(dim, -1)


def _idct(X, dim):
    X = X.transpose(dim, -1)
    N = X.shape[-1]
    X = X * math.sqrt(2.0 / N)
    X[..., 0] /= SQ2
    k = torch.arange(N, dtype=torch.float64, device=X.device)
    Xr = torch.cat([torch.zeros_like(X[..., :1]), X[..., 1:].flip(-1)], -1)
    V = torch.complex(X, -Xr) * torch.polar(torch.ones_like(k), math.pi * k / (2 * N))
    V[..., 0] *= 2
    v = torch.fft.ifft(V * (N / 2.0))
    x = torch.empty_like(X)
    x[..., ::2], x[..., 1::2] = v.real[..., :(N + 1) // 2], v.real[..., (N + 1) // 2:].flip(-1)
    return x.transpose(dim, -1)


def _dct2(x):
    return _dct(_dct(x, -1), -2)


def _idct2(x):
    return _idct(_idct(x, -1), -2)


def _eigs(N, h, bc):
    k = torch.arange(N, dtype=torch.float64, device=_dev())
    a = {"neumann": math.pi * k / (2 * N), "dirichlet": math.pi * (k + 1) / (2 * N), "periodic": math.pi * k / N}[bc]
    s = 4.0 / (h * h) * torch.sin(a) ** 2
    return s[:, None] + s[None, :]


def _elliptic(f, coef, h, bc):
    N = f.shape[-1]
    s = _eigs(N, h, bc)
    d = coef[0] + s * (coef[1] + coef[2] * s)
    if bc == "periodic":
        return torch.fft.ifft2(torch.fft.fft2(f) / d).real
    if bc == "neumann":
        return _idct2(_dct2(f) / d)
    i = torch.arange(N, device=f.device) % 2
    sign = (1 - 2 * ((i[:, None] + i[None, :]) % 2)).double()
    return sign * _idct2((_dct2(sign * f).flip(0, 1) / d).flip(0, 1))


def _ghost(u):
    return torch.nn.functional.pad(u[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]


def _faces(u, h):
    """East-west and north-south face differences, boundary faces included (zero there)."""
    g = _ghost(u)
    return (g[1:-1, 1:] - g[1:-1, :-1]) / h, (g[1:, 1:-1] - g[:-1, 1:-1]) / h


def _means(u):
    g = _ghost(u)
    return 0.5 * (g[1:-1, 1:] + g[1:-1, :-1]), 0.5 * (g[1:, 1:-1] + g[:-1, 1:-1])


def _div(fx, fy, h):
    return (fx[:, 1:] - fx[:, :-1]) / h + (fy[1:, :] - fy[:-1, :]) / h


def _reference_run(phi, psi, p, steps, scheme):
    """The MSAV step (BDF1 start, then BDF2) in physical space, as the scheme is written down."""
    N = phi.shape[-1]
    h = p.L / N
    ip = lambda a, b: h * h * (a * b).sum()
    lap = lambda u: _div(*_faces(u, h), h)
    mob = lambda u: [1.0 - p.M0 * (a * a - 1.0) ** 2 for a in _means(u)]

    def terms(f, c):
        pp, f2, f3 = torch.sin(0.5 * math.pi * f), f * f, f ** 3 - f
        fx, fy = _faces(f, h)
        gx, gy = fx * fx, fy * fy
        gbar = 0.5 * (gx[:, 1:] + gx[:, :-1]) + 0.5 * (gy[1:, :] + gy[:-1, :])
        fin = 0.5 * p.gamma_in * (c - p.psi_in) ** 2 + p.beta_in
        fout = 0.5 * p.gamma_out * (c - p.psi_out) ** 2 + p.beta_out
        one = torch.ones_like(f)
        IV = ip((f2 - 1.0 - p.beta) ** 2 / (4.0 * p.eps), one)
        IW = ip(6.0 * f2 * gbar + f3 ** 2 / p.eps ** 2, one)
        IZ = ip((1 + pp) * fin + (1 - pp) * fout, one)
        ax, ay = _means(f2)
        S = f * (f2 - 1.0 - p.beta) / p.eps / (2.0 * IV.sqrt())
        H = 3 * SQ2 / 4 * (f3 / p.eps - p.eps * lap(f))
        Q = (6.0 * (f * gbar - _div(ax * fx, ay * fy, h)) + f3 * (3 * f2 - 1.0) / p.eps ** 2) / IW.sqrt()
        K = 0.5 * math.pi * torch.cos(0.5 * math.pi * f) * (fin - fout) / (2.0 * IZ.sqrt())
        P = (p.gamma_in * (1 + pp) * (c - p.psi_in) + p.gamma_out * (1 - pp) * (c - p.psi_out)) / (2.0 * IZ.sqrt())
        return IV, IW, IZ, S, H, Q, K, P

    IV, IW, IZ, *_ = terms(phi, psi)
    X = [IV.sqrt(), 0.0, IW.sqrt(), IZ.sqrt()]
    Xo = list(X)
    fo, co = phi, psi
    s = _eigs(N, h, "neumann")
    C2 = p.M_phi * (p.gamma_surf * 3 * SQ2 * p.eps / 4 + p.theta)
    C3 = p.M_phi * p.gamma_bend * 3 * SQ2 * p.eps / 8
    tt = p.theta + p.gamma_bend * 3 * SQ2 / (4 * p.eps)
    cc = [p.M_phi * p.gamma_surf * 3 * SQ2 / 2, p.M_phi * p.gamma_area,
          p.M_phi * p.gamma_bend * 3 * SQ2 / (8 * p.eps), p.M_phi]
    for n in range(steps):
        bdf1 = n == 0 or scheme == "bdf1"
        a = 1.0 / p.dt if bdf1 else 1.5 / p.dt
        fs, cs = (phi, psi) if bdf1 else (2 * phi - fo, 2 * psi - co)
        _, _, _, S, H, Q, K, P = terms(fs, cs)
        F = [S, H, Q, K]
        wf, wc = (-phi, -psi) if bdf1 else (-4 * phi + fo, -4 * psi + co)
        div = 1.0 if bdf1 else 3.0
        aX = [((X[q] if bdf1 else 4 * X[q] - Xo[q]) + ip(F[q], wf) + (ip(P, wc) if q == 3 else 0.0)) / div
              for q in range(4)]
        scale = p.dt if bdf1 else 2 * p.dt
        f = -wf / scale - p.M_phi * tt * lap(fs)
        for q in range(4):
            f = f - cc[q] * aX[q] * F[q]
        sig = a + p.M_phi * p.gamma_surf * 3 * SQ2 * p.beta / (4 * p.eps) + s * (C2 + C3 * s)
        tau = a + p.lam * s
        mx, my = mob(fs)
        flux = lambda u: _div(mx * _faces(u, h)[0], my * _faces(u, h)[1], h)
        LP = flux(P)
        if scheme == "classical":
            g = -wc / scale + flux(aX[3] * P - p.lam * cs)
            mean = float((mx[:, 1:-1].sum() + my[1:-1, :].sum()) / (2 * N * (N - 1)))
            pre = a + p.lam * mean * s
            ch = lambda r: _cg(lambda u: a * u - p.lam * flux(u), lambda u: _idct2(_dct2(u) / pre), r)
        else:
            g = -wc / scale - p.lam * lap(cs) + aX[3] * LP
            ch = lambda r: _idct2(_dct2(r) / tau)
        chi = lambda r: _idct2(_dct2(r) / sig)
        fh, gh, Lh = chi(f), ch(g), ch(LP)
        Fh = [chi(u) for u in F]
        sums = torch.stack([ip(F[i], u) for i in range(4) for u in Fh + [fh]] + [ip(P, Lh), ip(P, gh)]).cpu().numpy()
        A, b = np.eye(5), np.zeros(5)
        A[:4, :4] += sums[:20].reshape(4, 5)[:, :4] * np.array(cc)
        A[:4, 4] = cc[3] * sums[:20].reshape(4, 5)[:, 3]
        b[:4] = sums[:20].reshape(4, 5)[:, 4]
        A[4, 3], A[4, 4], b[4] = -sums[20], 1.0 - sums[20], sums[21]
        y = np.linalg.solve(A, b)
        new = fh
        for q, w in enumerate((y[0], y[1], y[2], y[3] + y[4])):
            new = new - cc[q] * float(w) * Fh[q]
        fo, co, Xo = phi, psi, X
        phi, psi = new, gh + float(y[3] + y[4]) * Lh
        X = [float(y[0] + aX[0]), float(y[1] + aX[1]), float(y[2] + aX[2]), float(y[3] + y[4] + aX[3])]
    return phi, psi


def _cg(A, pre, b):
    x = pre(b)
    r = b - A(x)
    z = pre(r)
    d, rz = z, float((r * z).sum())
    stop = 1e-14 * float(b.norm())
    for _ in range(100):
        if float(r.norm()) <= stop:
            break
        Ad = A(d)
        al = rz / float((d * Ad).sum())
        x, r = x + al * d, r - al * Ad
        z = pre(r)
        new = float((r * z).sum())
        d, rz = z + (new / rz) * d, new
    return x


def _reference_smooth(phi, case):
    a, h, bc = _smooth_args(case), 1.0 / case["N"], case["bc"]
    for _ in range(case["steps"]):
        g = (phi ** 3 - phi) / a["eps"]
        r = phi / a["dt"] + a["mobility"] * _div(*_faces(g, h), h)
        phi = _elliptic(r, [1.0 / a["dt"], 0.0, a["mobility"] * a["eps"]], h, bc)
    return phi.clamp(-1.0, 1.0)


def exact(case, seed):
    if case["kind"] == "solve":
        return _elliptic(_solve_rhs(case, seed).double(), _solve_coef(case), 1.0 / case["N"], case["bc"])
    if case["kind"] == "smooth":
        return _reference_smooth(_smooth_input(case, seed).double(), case)
    rounded = lambda f: f.to(_dtype(case["precision"])).double()
    if case["kind"] == "batch":
        got = [_reference_run(*map(rounded, _fields(N, _many(N), s, case["column"])), _params(N, case), case["steps"], "cc")
               for N, s in _batch_members(case, seed)]
        return {f: torch.cat([g[i].reshape(-1).cpu() for g in got]) for i, f in enumerate(("phi", "psi"))}
    phi, psi = _reference_run(*map(rounded, _fields(case["N"], case["vesicles"], seed, case["column"])),
                              _params(case["N"], case), case["steps"], case["scheme"])
    res = {"phi": phi.cpu(), "psi": psi.cpu()}
    if case["energy"]:
        res["energy"] = None
    return res
