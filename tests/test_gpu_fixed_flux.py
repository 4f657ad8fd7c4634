"""The fixed-point Rusanov flux of the interface kernels (csrc/ader_fixr.cuh) where it
can go wrong: jumps at the faces from none (FP32 speed) through small ones (speed
refined in integers) to large ones (the FP64 form), gas at rest with power-of-two
pressure (carries in the conversion back), slow flow, other units, and the adiabatic
index.  Bar: the 1e-12 per step of the FP64 path, every variable by its own scale."""
import numpy as np
import pytest

import test_gpu_2d as t2
import test_gpu_3d as t3
import workloads as W
from test_gpu_dg import field_nonlinear, make, to_dev
from test_gpu_fixed_nd import worst

pytestmark = pytest.mark.gpu

CASES = [(1, N) for N in range(1, 8)] + [(2, N) for N in (1, 3, 5, 7)] + [(3, N) for N in (1, 3, 5)]
DIMS = {1: (67,), 2: (5, 7), 3: (3, 2, 5)}


def run(cuda, oracle_mod, D, N, change, gamma=1.4):
    import torch
    dims = DIMS[D]
    nc, h = int(np.prod(dims)), tuple(1.0 / d for d in dims)
    if D == 1:
        o = oracle_mod.Oracle(N, gamma=gamma)
        u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
        dt_of = lambda v: o.dg_dt(v, h[0])
        step = lambda v, dt: o.dg_step(v, h[0], dt)[0]
        ctx = make(cuda, nc, N, gamma=gamma)
    elif D == 2:
        o = oracle_mod.Oracle2D(N, gamma=gamma)
        u = np.array(t2.smooth_state(o, *dims, seed=N))
        dt_of = lambda v: o.dt(v, *dims, *h)
        step = lambda v, dt: o.step(v, *dims, *h, dt)[0]
        ctx = t2.make(*dims, N, gamma=gamma)
    else:
        o = oracle_mod.Oracle3D(N, gamma=gamma)
        u = np.array(t3.smooth_state(o, dims, (1.0,) * 3, seed=N))
        dt_of = lambda v: o.dt(v, dims, h)
        step = lambda v, dt: o.step(v, dims, h, dt)[0]
        ctx = t3.make(dims, N, gamma=gamma)
    shape = u.shape
    v = u.reshape(nc, (N + 1) ** D, D + 2).copy()
    change(v)
    v = v.reshape(shape)
    dt = 0.5 * dt_of(v)
    ud = to_dev(v, cuda)
    out = torch.empty_like(ud)
    ctx.ader_step(ud, out, dt)
    torch.cuda.synchronize()
    assert worst(out.cpu().numpy().reshape(shape), step(v, dt)) < 1e-12


@pytest.mark.parametrize("D,N", CASES)
@pytest.mark.parametrize("jump", [0.0, 1e-13, 1e-9, 1e-6, 1e-3, 0.5, 30.0])
def test_jumps(cuda, oracle_mod, D, N, jump):
    def change(v):  # cells scaled against one another: rho, then velocity, then energy
        g = np.random.default_rng(N + 10 * D)
        f = (1.0 + jump) ** g.uniform(-1, 1, (3, len(v), 1))
        v[..., 0] *= f[0]
        v[..., 1:-1] *= (f[0] * np.sqrt(f[1]))[..., None]
        v[..., -1] *= f[0] * f[1]
    run(cuda, oracle_mod, D, N, change)


@pytest.mark.parametrize("D,N", CASES)
@pytest.mark.parametrize("kind", ["rest", "slow", "light"])
def test_states(cuda, oracle_mod, D, N, kind):
    def change(v):
        if kind == "rest":
            v[..., 0], v[..., 1:-1] = 1.0, 0.0
            v[..., -1] = np.where(np.arange(len(v)) % 5 < 2, 2.5, 0.3125)[:, None]
        elif kind == "slow":  # Mach 1e-7, one direction only in some cells
            v[..., 1:-1] *= 1e-7
            v[::3, :, 1] = 0.0
        else:
            v[..., 0] *= 1e-5
            v[..., 1:-1] *= 1e-5 * 3e3
            v[..., -1] *= 1e-5 * 9e6
    run(cuda, oracle_mod, D, N, change)


@pytest.mark.parametrize("D,N", [(1, 4), (2, 3), (3, 2)])
@pytest.mark.parametrize("gamma", [1.05, 5.0 / 3.0, 2.0, 2.5])
def test_adiabatic_index(cuda, oracle_mod, D, N, gamma):
    """gamma - 1 above 1 takes the FP64 form"""
    run(cuda, oracle_mod, D, N, lambda v: None, gamma=gamma)


@pytest.mark.parametrize("system", ["reacting", "tracer"])
@pytest.mark.parametrize("N", [1, 3, 5, 7])
@pytest.mark.parametrize("what", ["all", "others", "none"])
@pytest.mark.parametrize("jump", [1e-14, 1e-11, 1e-9, 1e-6, 1e-2, 10.0])
def test_systems_jumps(cuda, oracle_mod, system, N, what, jump):
    """jumps of the further variables alone (their own bound on the wave speed's error and
    the path mean of u) and together with the Euler ones"""
    import test_gpu_fixed_systems as fs
    nc = 67
    o = oracle_mod.ReactingOracle(N, omega=1.0) if system == "reacting" else oracle_mod.NCOracle(N)
    u = (fs.reacting if system == "reacting" else fs.tracer)(o, nc, N)
    g = np.random.default_rng(N)
    f = (1.0 + jump) ** g.uniform(-1, 1, (4, nc, 1))
    if what == "all":
        u[..., 0] *= f[0]
        u[..., 1] *= f[0] * np.sqrt(f[1])
        u[..., 2] *= f[0] * f[1]
    if what != "none":
        for r in range(3, u.shape[-1]):
            u[..., r] *= f[r - 1]
    # (the wave speed is the Euler part's)
    dt = 0.5 * oracle_mod.Oracle(N).dg_dt(np.ascontiguousarray(u[..., :3]), 1.0 / nc)
    got, _ = fs.gpu_step(u, N, dt, system, **({"omega": 1.0} if system == "reacting" else {}))
    step = o.dg_step if system == "reacting" else o.step
    assert fs.worst(got, step(u, 1.0 / nc, dt)[0]) < 1e-12
