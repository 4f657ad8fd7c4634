"""The fixed-point form of the FP64 predictor (csrc/ader_fix.cuh) where it can go
wrong: meshes around its warp and block sizes, physical units far from one, time
steps far below the CFL step, cells of very different sizes side by side, and cells
that it hands to the FP64 tile code (jumps inside a cell, non-finite data).

Bar: the 1e-12 per step of the FP64 path, here for every variable by its own maximum
in the cell (the form keeps 57 bits below each cell's maxima)."""
import numpy as np
import pytest

import workloads as W
from test_gpu_dg import field_nonlinear, make, to_dev

pytestmark = pytest.mark.gpu


def predict(cuda, u, N, dt, x1=1.0, **kw):
    import torch
    ctx = make(cuda, u.shape[0], N, x1=x1, **kw)
    q = torch.empty(ctx.predictor_count, dtype=torch.float64, device=cuda)
    ctx.ader_predict(to_dev(u, cuda), dt, q)
    torch.cuda.synchronize()
    return q.cpu().numpy().reshape(u.shape[0], N + 1, N + 1, 3), ctx.ader_get_stats()


def per_cell_error(a, b):
    """largest |a - b| over a cell and variable, relative to that variable's scale in the cell
    (for m: sqrt(rho E), the flow's momentum unit)"""
    s = np.abs(b).max(axis=(1, 2))
    s[:, 1] = np.maximum(s[:, 1], np.sqrt(s[:, 0] * s[:, 2]))
    return float((np.abs(a - b).max(axis=(1, 2)) / s).max())


@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("cells", ["1", "warp-1", "warp+1", "block", "block+1", "many"])
def test_sizes(cuda, oracle_mod, N, cells):
    import torch
    warp = 32 // (N + 1)
    nc = {"1": 1, "warp-1": warp - 1, "warp+1": warp + 1, "block": 4 * warp,
          "block+1": 4 * warp + 1, "many": 152 * 24 * warp + 3}[cells]
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dt = o.dg_dt(u, 1.0 / nc)
    if cells == "many":  # past one round of resident blocks: a few cells of it
        ctx = make(cuda, nc, N)
        out = torch.empty(ctx.state_count, dtype=torch.float64, device=cuda)
        ctx.ader_step(to_dev(u, cuda), out, dt)
        at = np.array([0, 1, nc // 2, nc - 5 * warp, nc - 2, nc - 1])
        ref, _ = o.dg_step_cells(u, 1.0 / nc, dt, at)
        got = out.cpu().numpy().reshape(nc, -1)[at]
        assert np.abs(got - ref.reshape(len(at), -1)).max() < 1e-12 * np.abs(ref).max()
        assert ctx.ader_get_stats()["cells"] == nc
        return
    ref, iters = o.predict(u, dt * nc)
    q, st = predict(cuda, u, N, dt)
    assert per_cell_error(q, ref) < 1e-12
    assert st["cells"] == nc and abs(st["max_iters"] - iters.max()) <= 1


@pytest.mark.parametrize("N", [1, 2, 5, 7])
@pytest.mark.parametrize("rho,vel", [(1.2, 340.0), (1e-6, 3e4), (8e3, 0.01), (1e12, 1.0)])
def test_units(cuda, oracle_mod, N, rho, vel):
    """the same flow in other units; the last density is outside the form's scales"""
    nc = 23
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(3 + N), o.node_x(nc)) * rho * vel ** np.arange(3)
    dt = o.dg_dt(u, 1.0 / nc)
    o.set(fixed_iter=N + 2)
    ref, _ = o.predict(u, dt * nc)
    q, _ = predict(cuda, u, N, dt, picard_fixed_iter=N + 2)
    assert per_cell_error(q, ref) < 1e-12


@pytest.mark.parametrize("N", [1, 3, 5, 7])
@pytest.mark.parametrize("factor", [1e-1, 1e-3, 1e-7, 1e-12])
def test_small_time_steps(cuda, oracle_mod, N, factor):
    """the last step of a solve can be any fraction of the CFL step"""
    nc = 37
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dt = factor * o.dg_dt(u, 1.0 / nc)
    ref, _ = o.predict(u, dt * nc)
    q, _ = predict(cuda, u, N, dt)
    assert per_cell_error(q, ref) < 1e-12


@pytest.mark.parametrize("N", [1, 2, 4, 5, 7])
@pytest.mark.parametrize("ratio", [3.0, 40.0, 1e4, 1e9])
def test_uneven_cells(cuda, oracle_mod, N, ratio):
    """neighbouring cells (of one warp) whose density and pressure differ by `ratio`: every cell
    has its own units, the table of kappa~ is the warp's"""
    nc = 29
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    g = np.random.default_rng(N)
    a, b = (ratio ** g.uniform(-1, 0, nc) for _ in range(2))
    u[..., 0] *= a[:, None]
    u[..., 1] *= np.sqrt(a * b)[:, None]
    u[..., 2] *= b[:, None]
    dt = o.dg_dt(u, 1.0 / nc)
    o.set(fixed_iter=4)
    ref, _ = o.predict(u, dt * nc)
    q, _ = predict(cuda, u, N, dt, picard_fixed_iter=4)
    assert per_cell_error(q, ref) < 1e-12


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("bad", ["density", "pressure", "negative", "nan", "inf"])
def test_redone_cells(cuda, oracle_mod, N, bad):
    """cells outside the form's range: they equal the oracle's FP64 result, and the others are
    what they are without them"""
    nc = 61
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dt = 0.2 * o.dg_dt(u, 1.0 / nc)
    at = [0, 7, 8, nc - 1]
    v = u.copy()
    n = N + 1
    step = np.where(np.arange(n) < n // 2, 1.0, 0.01)
    for c in at:
        if bad == "density":
            v[c, :, 0] *= step
            v[c, :, 1] *= step
            v[c, :, 2] -= 0.5 * u[c, :, 1] ** 2 / u[c, :, 0] * (1 - step)
        elif bad == "pressure":
            v[c, :, 2] *= np.where(np.arange(n) < n // 2, 1.0, 60.0)
        elif bad == "negative":
            v[c, 0, 0] = -0.3
        elif bad == "nan":
            v[c, n - 1, 1] = np.nan
        else:
            v[c, 0, 2] = np.inf
    o.set(fixed_iter=3)
    ref, _ = o.predict(v, dt * nc)
    q, st = predict(cuda, v, N, dt, picard_fixed_iter=3)
    q0, _ = predict(cuda, u, N, dt, picard_fixed_iter=3)
    rest = np.setdiff1d(np.arange(nc), at)
    assert np.array_equal(q[rest], q0[rest])
    assert st["cells"] == nc
    if bad in ("nan", "inf"):
        assert not np.isfinite(q[at]).all(axis=(1, 2, 3)).any()
    else:
        assert per_cell_error(q[at], ref[at]) < 1e-12


@pytest.mark.parametrize("gamma", [1.1, 5.0 / 3.0, 2.0, 2.5])
def test_adiabatic_index(cuda, oracle_mod, gamma):
    """gamma - 1 above 1 takes the FP64 kernel"""
    nc, N = 31, 4
    o = oracle_mod.Oracle(N, gamma=gamma)
    u = W.nodal_state(field_nonlinear(2), o.node_x(nc))
    dt = o.dg_dt(u, 1.0 / nc)
    ref, _ = o.predict(u, dt * nc)
    q, _ = predict(cuda, u, N, dt, gamma=gamma)
    assert per_cell_error(q, ref) < 1e-12


def test_iteration_cap_and_tight_tolerance(cuda, oracle_mod):
    from paper_2409_12483_gb300 import capi
    nc, N = 40, 3
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(1), o.node_x(nc))
    dt = o.dg_dt(u, 1.0 / nc)
    _, st = predict(cuda, u, N, dt, picard_max_iter=2)
    assert st["max_iters"] == 2 and st["status"] == capi.ADER_ERR_NOT_CONVERGED
    o.set(tol=1e-3)
    ref, iters = o.predict(u, dt * nc)
    q, st = predict(cuda, u, N, dt, picard_tol=1e-3)
    assert st["max_iters"] == iters.max() and per_cell_error(q, ref) < 1e-12
