"""The limiter's cell list (csrc/ader_limiter.cuh) where it can go wrong: meshes around
the detector blocks (126 cells), warps whose undecided cells are few (decided by the
recomputing blocks) or many (decided in place; strict NAD in constant regions), both
boundary conditions, and steps that follow one another (the list starts empty).
Bar: the oracle's flags exactly and 1e-12 per step, as the limiter's other tests."""
import numpy as np
import pytest

from conftest import rel_linf
from test_gpu_dg import to_dev
from test_gpu_limiter import make
from test_oracle_limiter import conserved

pytestmark = pytest.mark.gpu


def tube(o, nc, bumps):
    """pressure jumps on cell faces, and gas at rest or (bumps) waves everywhere"""
    x = o.node_x(nc)
    wave = 0.2 * np.sin(2 * np.pi * 7 * x) if bumps else np.zeros(x.shape)
    left = (x * nc > nc // 3) & (x * nc < 2 * nc // 3)
    return conserved(np.where(left, 1.0, 0.125) * (1 + wave), wave, np.where(left, 1.0, 0.1))


@pytest.mark.parametrize("nc", [3, 31, 125, 126, 127, 253])
@pytest.mark.parametrize("N", [1, 2, 3, 5, 7])
@pytest.mark.parametrize("strict,bumps,bc", [(True, False, "outflow"), (True, True, "periodic"),
                                             (False, False, "periodic")])
def test_listed_cells(cuda, oracle_mod, N, nc, strict, bumps, bc):
    import torch
    o = oracle_mod.Oracle(N)
    nad = dict(delta0=0.0, eps=0.0) if strict else {}
    u = tube(o, nc, bumps)
    dx = 1.0 / nc
    dt = o.dg_dt(u, dx)
    ref, tr, rc = o.dgl_step(u, dx, dt, bc=bc, limiter=True, **nad)
    assert rc == 0
    ctx = make(nc, N, bc=bc, limiter=1, **{"nad_" + k: v for k, v in nad.items()})
    ud = to_dev(u, cuda)
    out = torch.empty_like(ud)
    for _ in range(2):  # the same step twice: the second starts from an empty list
        ctx.ader_step(ud, out, dt)
        flags = ctx.ader_get_troubled().cpu().numpy()
        torch.cuda.synchronize()
        # rounding of P u* where the state is constant decides the strict principle there
        flat = (np.ptp(u.reshape(nc, -1, 3), axis=1) == 0).all(1) & strict & (not bumps)
        flat &= np.roll(flat, 1) & np.roll(flat, -1)
        np.testing.assert_array_equal(flags[~flat], tr[~flat])
        near = flat | np.roll(flat, 1) | np.roll(flat, -1)
        got = out.cpu().numpy().reshape(nc, -1)
        assert rel_linf(got[~near], ref.reshape(nc, -1)[~near]) < 1e-12 if (~near).any() else True
        assert rel_linf(got, ref.reshape(nc, -1)) < 1e-10
        assert ctx.ader_get_stats()["troubled_cells"] == flags.sum()


def test_two_steps_list_their_own_cells(cuda, oracle_mod):
    import torch
    N, nc = 3, 130
    o = oracle_mod.Oracle(N)
    u = tube(o, nc, False)
    ref, steps, _, rc, total = o.dgl_solve(u, 1.0 / nc, max_steps=12, limiter=True)
    assert rc == 0
    ctx = make(nc, N, limiter=1)
    ud = to_dev(u, cuda)
    assert ctx.ader_solve(ud, max_steps=12)[0] == steps
    torch.cuda.synchronize()
    assert ctx.ader_get_stats()["troubled_cells"] == total > 0
    assert rel_linf(ud.cpu().numpy(), ref) < 1e-11
