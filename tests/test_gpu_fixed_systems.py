"""The fixed-point form of the nested predictors (csrc/ader_fixs.cuh: reacting and
tracer systems) where it can go wrong: meshes around its warp and block sizes, further
variables of other sizes than the Euler ones, reaction frequencies, time steps far below
the CFL step, and cells handed to the FP64 tile code.

Bar: 1e-12 per step; every variable by its own scale, which is at least a tenth of the
largest one's because both sides iterate to 1e-13 of the whole state."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def reacting(o, nc, seed=0, c1=1.0, c2=1.0):
    u = W.reacting_state(o.node_x(nc), seed=seed)
    u[..., 3] *= c1
    u[..., 4] *= c2
    return u


def tracer(o, nc, seed=0, a=1.0):
    x = o.node_x(nc)
    u = W.reacting_state(x, seed=seed)[..., :4].copy()
    u[..., 3] = a * np.sin(2 * np.pi * x + seed)
    return u


def gpu_step(u, N, dt, system, **kw):
    import torch
    from paper_2409_12483_gb300 import Context
    ctx = Context(u.shape[0], N, "dg", system=system, **kw)
    ud = torch.tensor(u.reshape(-1), device="cuda")
    out = torch.empty_like(ud)
    ctx.ader_step(ud, out, dt)
    torch.cuda.synchronize()
    return out.cpu().numpy().reshape(u.shape), ctx.ader_get_stats()


def worst(a, ref):
    M = a.shape[-1]
    a, ref = a.reshape(-1, M), ref.reshape(-1, M)
    s = np.abs(ref).max(0)
    s = np.maximum(s, 0.1 * max(1.0, s.max()))
    return float((np.abs(a - ref).max(0) / s).max())


@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("cells", ["1", "warp-1", "warp+1", "block+1"])
def test_sizes(cuda, oracle_mod, N, cells):
    warp = 32 // (N + 1)
    nc = {"1": 1, "warp-1": warp - 1, "warp+1": warp + 1, "block+1": 4 * warp + 1}[cells]
    o = oracle_mod.ReactingOracle(N, omega=2.0)
    u = reacting(o, nc, N)
    dt = o.dg_dt(u, 1.0 / nc)
    got, st = gpu_step(u, N, dt, "reacting", omega=2.0)
    assert worst(got, o.dg_step(u, 1.0 / nc, dt)[0]) < 1e-12 and st["cells"] == nc
    o = oracle_mod.NCOracle(N)
    u = tracer(o, nc, N)
    dt = o.dt(u, 1.0 / nc)
    got, st = gpu_step(u, N, dt, "tracer")
    assert worst(got, o.step(u, 1.0 / nc, dt)[0]) < 1e-12 and st["cells"] == nc


@pytest.mark.parametrize("N", [2, 5])
def test_more_tiles_than_resident_blocks(cuda, oracle_mod, N):
    """a few cells of a mesh whose blocks take several tiles each"""
    warp = 32 // (N + 1)
    nc = 152 * 5 * 4 * warp * 2 + 3
    o = oracle_mod.ReactingOracle(N, omega=2.0)
    u = reacting(o, nc, N)
    dt = o.dg_dt(u, 1.0 / nc)
    got, st = gpu_step(u, N, dt, "reacting", omega=2.0)
    at = np.array([0, 1, nc // 3, nc - 4 * warp, nc - 1])
    ref, _ = o.dg_step_cells(u, 1.0 / nc, dt, at)
    assert worst(got[at], ref) < 1e-12 and st["cells"] == nc


@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("c1,c2", [(1e-4, 3.0), (1e3, 1e-2), (0.0, 0.0), (1.0, 0.0), (-1.0, 1e-9)])
@pytest.mark.parametrize("omega", [0.0, 30.0])
def test_species_scales(cuda, oracle_mod, N, c1, c2, omega):
    nc = 33
    o = oracle_mod.ReactingOracle(N, omega=omega)
    u = reacting(o, nc, 3, c1, c2)
    dt = o.dg_dt(u, 1.0 / nc)
    got, _ = gpu_step(u, N, dt, "reacting", omega=omega)
    assert worst(got, o.dg_step(u, 1.0 / nc, dt)[0]) < 1e-12


@pytest.mark.parametrize("N", [1, 3, 6])
@pytest.mark.parametrize("a", [0.0, 1e-6, 1.0, 1e5, 1e15])
@pytest.mark.parametrize("factor", [1.0, 1e-6])
def test_tracer_scales_and_small_time_steps(cuda, oracle_mod, N, a, factor):
    nc = 33
    o = oracle_mod.NCOracle(N)
    u = tracer(o, nc, 2, a)
    dt = factor * o.dt(u, 1.0 / nc)
    got, _ = gpu_step(u, N, dt, "tracer")
    assert worst(got, o.step(u, 1.0 / nc, dt)[0]) < 1e-12


@pytest.mark.parametrize("N", [1, 2, 5, 7])
@pytest.mark.parametrize("system", ["reacting", "tracer"])
def test_redone_cells(cuda, oracle_mod, N, system):
    """cells with a density jump or a NaN inside; the others are what they are without them"""
    nc, n = 41, N + 1
    o = oracle_mod.ReactingOracle(N, omega=2.0) if system == "reacting" else oracle_mod.NCOracle(N)
    u = reacting(o, nc, 1) if system == "reacting" else tracer(o, nc, 1)
    dt = 0.1 * (o.dg_dt(u, 1.0 / nc) if system == "reacting" else o.dt(u, 1.0 / nc))
    kw = {"omega": 2.0} if system == "reacting" else {}
    clean, _ = gpu_step(u, N, dt, system, **kw)
    v = u.copy()
    low = np.arange(n) >= n // 2
    v[5, low, 0] *= 0.11
    v[5, low, 1] *= 0.11
    v[30, 0, 3] = np.nan
    got, st = gpu_step(v, N, dt, system, **kw)
    assert st["cells"] == nc
    v[30] = u[30]
    ref = (o.dg_step(v, 1.0 / nc, dt)[0] if system == "reacting" else o.step(v, 1.0 / nc, dt)[0]
           ).reshape(u.shape)
    fine = np.isfinite(ref).all((1, 2))
    fine[29:32] = False
    assert fine.sum() >= nc - 6
    assert worst(got[fine], ref[fine]) < 1e-12
    rest = np.setdiff1d(np.arange(nc), [4, 5, 6, 29, 30, 31])
    assert np.array_equal(got[rest], clean[rest])
    assert not np.isfinite(got[30]).all()
