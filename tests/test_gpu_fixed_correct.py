"""The corrector on a given space-time state (ader_correct) in fixed point: its epilogue
(csrc/ader_fix.cuh) on states that the predictor made, on states of other sizes than u, on
states outside the form's range (handed to the FP64 tile code) and on non-finite ones.
Bar: 1e-12 per step, every variable by its own scale."""
import numpy as np
import pytest

import workloads as W
from test_gpu_dg import field_nonlinear, make, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", range(1, 8))
@pytest.mark.parametrize("nc", [3, 31, 67])
def test_predict_then_correct_is_a_step(cuda, oracle_mod, N, nc):
    import torch
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dt = o.dg_dt(u, 1.0 / nc)
    ctx = make(cuda, nc, N)
    ud = to_dev(u, cuda)
    q = torch.empty(ctx.predictor_count, dtype=torch.float64, device=cuda)
    out, ref = torch.empty_like(ud), torch.empty_like(ud)
    ctx.ader_predict(ud, dt, q)
    ctx.ader_correct(ud, q, dt, out)
    ctx.ader_step(ud, ref, dt)
    torch.cuda.synchronize()
    a, b = out.cpu().numpy().reshape(-1, 3), o.dg_step(u, 1.0 / nc, dt)[0].reshape(-1, 3)
    assert (np.abs(a - b).max(0) < 1e-12 * np.abs(b).max(0)).all()
    c = ref.cpu().numpy().reshape(-1, 3)
    assert (np.abs(a - c).max(0) < 1e-13 * np.abs(c).max(0)).all()


@pytest.mark.parametrize("N", [1, 3, 5, 7])
@pytest.mark.parametrize("kind", ["scaled", "light node", "nan", "gamma"])
def test_given_states(cuda, oracle_mod, N, kind):
    """against the corrector by dense sums in numpy (bar times the sums' n^2 terms)"""
    import torch
    nc, n = 41, N + 1
    o = oracle_mod.Oracle(N)
    u = W.nodal_state(field_nonlinear(N), o.node_x(nc))
    dt = o.dg_dt(u, 1.0 / nc)
    gamma = 1.4 if kind != "gamma" else 5.0 / 3.0
    oo = oracle_mod.Oracle(N, gamma=gamma)
    q = np.array(oo.predict(u, dt * nc)[0]).reshape(nc, n, n, 3)
    bad = np.zeros(nc, bool)
    if kind == "scaled":
        q = q * np.array([3.7, 0.2, 11.0])
    elif kind == "light node":  # density down to 1/64 of the cell's largest
        bad[[0, nc // 2]] = True
        q[bad, 0, 0] *= np.array([1 / 64, 1 / 64, 1 / 64])
    elif kind == "nan":
        q[nc // 3, 0, 0, 2] = np.nan
    ctx = make(cuda, nc, N, gamma=gamma)
    ud = to_dev(u, cuda)
    out = torch.empty_like(ud)
    ctx.ader_correct(ud, to_dev(q, cuda), dt, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy().reshape(nc, n, 3)
    # the corrector by dense sums in numpy
    w, Dt = o.table("w"), o.table("dt_m")
    psi0, psi1 = o.table("psi0"), o.table("psi1")

    def flux(U):
        vel = U[..., 1] / U[..., 0]
        p = (gamma - 1) * (U[..., 2] - 0.5 * U[..., 1] * vel)
        return np.stack([U[..., 1], U[..., 1] * vel + p, (U[..., 2] + p) * vel], -1), vel, p

    lam = dt * nc
    F, _, _ = flux(q)
    vol = u.reshape(nc, n, 3) + lam * np.einsum("kl,clr->ckr", Dt, np.einsum("t,ctlr->clr", w, F)) / w[:, None]
    a, b = np.einsum("l,ctlr->ctr", psi1, q), np.roll(np.einsum("l,ctlr->ctr", psi0, q), -1, 0)
    (Fa, va, pa), (Fb, vb, pb) = flux(a), flux(b)
    with np.errstate(invalid="ignore"):
        s = np.maximum(abs(va) + np.sqrt(gamma * pa / a[..., 0]), abs(vb) + np.sqrt(gamma * pb / b[..., 0]))
    # (a trace that is not physical makes the flux NaN)
    s[(a[..., 0] <= 0) | (pa <= 0) | (b[..., 0] <= 0) | (pb <= 0)] = np.nan
    G = lam * np.einsum("t,ctr->cr", w, 0.5 * (Fa + Fb) - 0.5 * s[..., None] * (b - a))
    ref = vol - (psi1[:, None] * G[:, None] - psi0[:, None] * np.roll(G, 1, 0)[:, None]) / w[:, None]
    fine = np.isfinite(ref).all((1, 2))
    assert np.array_equal(fine, np.isfinite(got).all((1, 2))) and fine.any()
    scale = np.abs(ref[fine]).max((0, 1))
    scale[1] = max(scale[1], np.sqrt(scale[0] * scale[2]))
    assert (np.abs(got[fine] - ref[fine]).max((0, 1)) < 1e-12 * scale * n * n).all()
