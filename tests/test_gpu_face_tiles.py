"""The interface kernel's tiles (the cells between 32 or 64 faces): meshes around the
tile sizes, one- and two-pass blocks, both schemes and both boundary conditions.
Bar: 1e-12 per step against the oracle, and lambda_max of the new state exactly the
oracle's time step (1e-13)."""
import numpy as np
import pytest

import workloads as W
from conftest import rel_linf
from test_gpu_dg import field_nonlinear, make, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [1, 2, 30, 31, 32, 62, 63, 64, 65, 127])
@pytest.mark.parametrize("faces", [32, 64])
@pytest.mark.parametrize("N", [0, 2, 3, 4, 5, 7])
def test_dg_tiles(cuda, oracle_mod, N, faces, nc):
    import torch
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dx = 1.0 / nc
    ctx = make(cuda, nc, N)
    ctx.ader_set_tuning(face_cells_per_block=faces)
    ud = to_dev(u, cuda)
    steps, t, _ = ctx.ader_solve(ud, max_steps=3)
    torch.cuda.synchronize()
    ref, tr = u, 0.0
    for _ in range(3):
        dt = o.dg_dt(ref, dx)
        ref, tr = o.dg_step(ref, dx, dt)[0], tr + dt
    assert steps == 3 and abs(t - tr) < 1e-13 * tr
    assert rel_linf(ud.cpu().numpy().reshape(ref.shape), ref) < 3e-12


@pytest.mark.parametrize("nc", [31, 32, 63, 64, 127])
@pytest.mark.parametrize("faces", [32, 64])
@pytest.mark.parametrize("N", [2, 4])
def test_fv_and_outflow_tiles(cuda, oracle_mod, N, faces, nc):
    import torch
    from paper_2409_12483_gb300 import Context
    o = oracle_mod.Oracle(N)
    dx = 1.0 / nc
    v = W.cell_average_state(field_nonlinear(3), nc)
    ctx = Context(nc, N, "fv")
    ctx.ader_set_tuning(face_cells_per_block=faces)
    vd, out = to_dev(v, cuda), torch.empty(v.size, dtype=torch.float64, device=cuda)
    dt = o.fv_dt(v, dx)
    ctx.ader_step(vd, out, dt)
    torch.cuda.synchronize()
    assert rel_linf(out.cpu().numpy().reshape(v.shape), o.fv_step(v, dx, dt)[0]) < 1e-12
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dt = o.dg_dt(u, dx)
    ref = o.dgl_step(u, dx, dt, bc="outflow", limiter=False)[0]
    ctx = make(cuda, nc, N, bc="outflow")
    ctx.ader_set_tuning(face_cells_per_block=faces)
    ud = to_dev(u, cuda)
    out = torch.empty_like(ud)
    ctx.ader_step(ud, out, dt)
    torch.cuda.synchronize()
    assert rel_linf(out.cpu().numpy().reshape(ref.shape), ref) < 1e-12
