"""One step at high Mach number, where the pressure is a small part of the energy and so of
the fixed-point form's unit: 1D, 2D, 3D and both systems with further variables, along the
faces' normals and across them.  Uniform velocity and, inside a cell, uniform pressure (so
that every trace has the pressure of its cell); jumps of density, velocity and pressure at
the faces.  Bar: the 1e-12 per step of the FP64 path, every variable by its own scale."""
import numpy as np
import pytest

import test_gpu_2d as t2
import test_gpu_3d as t3
from test_gpu_dg import make, to_dev
from test_gpu_fixed_nd import worst

pytestmark = pytest.mark.gpu

DIMS = {1: (67,), 2: (5, 7), 3: (3, 2, 5)}


def state(D, N, nc, mach, jump, way):
    """[cell][node][variable]; way: the velocity's direction"""
    g = np.random.default_rng(N + 10 * D)
    cell = lambda: (1 + jump * g.uniform(-1, 1, (nc, 1)))
    rho = cell() * (1 + 0.1 * g.uniform(-1, 1, (nc, (N + 1) ** D)))
    p = cell() * np.ones_like(rho)
    way = np.asarray(way, float) / np.linalg.norm(way)
    vel = [mach * np.sqrt(1.4) * w * cell() * np.ones_like(rho) for w in way]
    E = p / 0.4 + 0.5 * rho * sum(v * v for v in vel)
    return np.stack([rho, *(rho * v for v in vel), E], -1)


@pytest.mark.parametrize("D,N,slant", [(1, N, False) for N in (1, 3, 5, 7)] + [
    (D, N, slant) for D, N in [(2, 1), (2, 3), (2, 5), (3, 1), (3, 3)] for slant in (False, True)])
@pytest.mark.parametrize("jump", [1e-6, 1e-4, 1e-3])
@pytest.mark.parametrize("mach", [3.0, 30.0, 100.0, 1000.0])
def test_mach(cuda, oracle_mod, D, N, slant, jump, mach):
    import torch
    dims = DIMS[D]
    nc, h = int(np.prod(dims)), tuple(1.0 / d for d in dims)
    u = state(D, N, nc, mach, jump, [1.0] if D == 1 else [1e-3, 1.0, 0.3][:D] if slant
              else [1.0, 0.6, -0.8][:D])
    if D == 1:
        o, ctx = oracle_mod.Oracle(N), make(cuda, nc, N)
        dt = 0.5 * o.dg_dt(u, h[0])
        ref = o.dg_step(u, h[0], dt)[0]
    elif D == 2:
        o, ctx = oracle_mod.Oracle2D(N), t2.make(*dims, N)
        dt = 0.5 * o.dt(u, *dims, *h)
        ref = o.step(u, *dims, *h, dt)[0]
    else:
        o, ctx = oracle_mod.Oracle3D(N), t3.make(dims, N)
        dt = 0.5 * o.dt(u, dims, h)
        ref = o.step(u, dims, h, dt)[0]
    ud = to_dev(u, cuda)
    out = torch.empty_like(ud)
    ctx.ader_step(ud, out, dt)
    torch.cuda.synchronize()
    assert worst(out.cpu().numpy().reshape(u.shape), np.asarray(ref).reshape(u.shape)) < 1e-12


@pytest.mark.parametrize("system", ["reacting", "tracer"])
@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("jump", [1e-6, 1e-3])
@pytest.mark.parametrize("mach", [3.0, 100.0, 1000.0])
def test_mach_systems(cuda, oracle_mod, system, N, jump, mach):
    import test_gpu_fixed_systems as fs
    nc = 67
    u = state(1, N, nc, mach, jump, [1.0])
    g = np.random.default_rng(3)
    extra = 1 + 0.3 * g.uniform(-1, 1, (nc, 1, 2)) * np.ones((1, N + 1, 1))
    u = np.concatenate([u, extra[..., :2 if system == "reacting" else 1]], -1)
    o = oracle_mod.ReactingOracle(N, omega=1.0) if system == "reacting" else oracle_mod.NCOracle(N)
    dt = 0.5 * oracle_mod.Oracle(N).dg_dt(np.ascontiguousarray(u[..., :3]), 1.0 / nc)
    got, _ = fs.gpu_step(u, N, dt, system, **({"omega": 1.0} if system == "reacting" else {}))
    ref = (o.dg_step if system == "reacting" else o.step)(u, 1.0 / nc, dt)[0].reshape(u.shape)
    assert worst(got[..., :3], ref[..., :3]) < 1e-12
    s = np.abs(ref).max((0, 1))
    assert (np.abs(got - ref).max((0, 1))[3:] / s[3:]).max() < 1e-12
