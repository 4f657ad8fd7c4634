"""The fixed-point predictors give a cell the same bits whatever cells share its warp or
block: a mesh of ordinary cells with slow ones in between (sound and flow speeds down by
1e-2 to 1e-7, so that their share of the time step is far from the others') against the mesh
without them, and the slow cells against a mesh of slow cells only.  The split of a mesh over
several contexts relies on this."""
import numpy as np
import pytest

import test_gpu_2d as t2
import test_gpu_3d as t3
import workloads as W
from test_gpu_dg import field_nonlinear
from test_gpu_fixed import per_cell_error, predict

pytestmark = pytest.mark.gpu


def slowed(u, at, factor, D=1):
    v = u.copy()
    v[at, ..., 1:1 + D] *= factor
    v[at, ..., 1 + D] *= factor * factor
    return v


@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("factor", [1e-1, 1e-2, 1e-4, 1e-7])
def test_1d(cuda, oracle_mod, N, factor):
    nc = 4 * (32 // (N + 1)) + 3
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dt = o.dg_dt(u, 1.0 / nc)
    at = np.arange(1, nc, 3)
    rest = np.setdiff1d(np.arange(nc), at)
    mixed = slowed(u, at, factor)
    q, st = predict(cuda, mixed, N, dt, picard_fixed_iter=4)
    plain, _ = predict(cuda, u, N, dt, picard_fixed_iter=4)
    slow, _ = predict(cuda, slowed(u, np.arange(nc), factor), N, dt, picard_fixed_iter=4)
    assert np.array_equal(q[rest], plain[rest])
    assert np.array_equal(q[at], slow[at])
    o.set(fixed_iter=4)
    assert per_cell_error(q, o.predict(mixed, dt * nc)[0]) < 1e-12


@pytest.mark.parametrize("D,N", [(2, 1), (2, 2), (2, 3), (3, 1), (3, 2)])
@pytest.mark.parametrize("factor", [1e-2, 1e-5])
def test_nd(cuda, oracle_mod, D, N, factor):
    """a step; cells with no slow neighbour across a face, in meshes of two rows or planes (the
    cells of a block lie in one) of which only the second has the slow cells"""
    import torch
    dims = (40, 3) if D == 2 else (20, 3, 3)
    h = tuple(1.0 / d for d in dims)
    nc = int(np.prod(dims))
    o = (oracle_mod.Oracle2D if D == 2 else oracle_mod.Oracle3D)(N)
    u = np.array(t2.smooth_state(o, *dims, seed=N) if D == 2
                 else t3.smooth_state(o, dims, (1.0,) * 3, seed=N))
    dt = 0.5 * (o.dt(u, *dims, *h) if D == 2 else o.dt(u, dims, h))
    flat = u.reshape(nc, -1, D + 2)
    at = np.arange(3, nc, 9)
    row = np.arange(nc).reshape(dims[::-1])
    touched = np.isin(row, at)
    for ax in range(D):
        touched = touched | np.isin(np.roll(row, 1, ax), at) | np.isin(np.roll(row, -1, ax), at)
    rest = row[~touched]
    assert rest.size > nc // 8
    got = []
    for v in (flat, slowed(flat, at, factor, D)):
        ctx = (t2.make(*dims, N, picard_fixed_iter=4) if D == 2
               else t3.make(dims, N, picard_fixed_iter=4))
        ud = t2.to_dev(v)
        out = torch.empty_like(ud)
        ctx.ader_step(ud, out, dt)
        torch.cuda.synchronize()
        got.append(out.cpu().numpy().reshape(flat.shape))
    assert np.array_equal(got[0][rest], got[1][rest])


@pytest.mark.parametrize("system", ["reacting", "tracer"])
@pytest.mark.parametrize("N", [1, 3, 6])
@pytest.mark.parametrize("factor", [1e-2, 1e-5])
def test_systems(cuda, oracle_mod, system, N, factor):
    import test_gpu_fixed_systems as fs
    nc = 4 * (32 // (N + 1)) + 3
    o = oracle_mod.ReactingOracle(N, omega=2.0) if system == "reacting" else oracle_mod.NCOracle(N)
    u = (fs.reacting if system == "reacting" else fs.tracer)(o, nc, N)
    kw = {"omega": 2.0} if system == "reacting" else {}
    dt = 0.5 * (o.dg_dt(u, 1.0 / nc) if system == "reacting" else o.dt(u, 1.0 / nc))
    at = np.arange(2, nc - 1, 5)
    rest = np.setdiff1d(np.arange(nc), np.concatenate([at - 1, at, at + 1]))
    mixed = slowed(u, at, factor)
    plain, _ = fs.gpu_step(u, N, dt, system, **kw)
    got, _ = fs.gpu_step(mixed, N, dt, system, **kw)
    assert np.array_equal(got[rest], plain[rest])
    ref = (o.dg_step if system == "reacting" else o.step)(mixed, 1.0 / nc, dt)[0].reshape(u.shape)
    assert fs.worst(got, ref) < 1e-12


@pytest.mark.parametrize("N", [2, 5])
def test_shards(cuda, oracle_mod, N):
    """a mesh with a slow third, split where its halo does not line up with a warp's cells: the
    local cells are those of the single mesh bit for bit"""
    import torch
    from paper_2409_12483_gb300 import Context
    from paper_2409_12483_gb300.capi import ShardContext
    nc, first, nl = 97, 31, 34
    o = oracle_mod.Oracle(N)
    u = slowed(W.nodal_state(field_nonlinear(N), o.node_x(nc)), np.arange(40, 72), 1e-3)
    one = Context(nc, N, "dg")
    ud = torch.tensor(u.reshape(-1), device=cuda)
    dt = 0.5 * one.ader_compute_dt(ud)
    out = torch.empty_like(ud)
    one.ader_step(ud, out, dt)
    ctx = ShardContext(nc, first, nl, N, "dg")
    H = ctx.halo
    us = torch.tensor(np.ascontiguousarray(u[first - H:first + nl + H]).reshape(-1), device=cuda)
    outs = torch.empty_like(us)
    ctx.ader_step(us, outs, dt)
    torch.cuda.synchronize()
    whole = out.cpu().numpy().reshape(nc, -1)[first:first + nl]
    part = outs.cpu().numpy().reshape(nl + 2 * H, -1)[H:H + nl]
    assert np.array_equal(part, whole)
