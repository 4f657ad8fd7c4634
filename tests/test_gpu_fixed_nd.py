"""The fixed-point form of the 2D and 3D predictors (csrc/ader_fixd.cuh) where it can
go wrong: several cells per block and a partial last block, other units, time steps far
below the CFL step, neighbours of very different sizes, and cells handed to the FP64
block code.  Bar: 1e-12 per step against the oracle, every variable by its own scale."""
import numpy as np
import pytest

import test_gpu_2d as t2
import test_gpu_3d as t3

pytestmark = pytest.mark.gpu

CASES = [(2, N) for N in range(1, 8)] + [(3, N) for N in range(1, 5)]
DIMS = {2: (5, 7), 3: (3, 2, 5)}


def setup(oracle_mod, D, N):
    dims = DIMS[D]
    h = tuple(1.0 / d for d in dims)
    if D == 2:
        o = oracle_mod.Oracle2D(N)
        u = np.array(t2.smooth_state(o, *dims, seed=N))
        return o, u, dims, lambda v: o.dt(v, *dims, *h), lambda v, dt: o.step(v, *dims, *h, dt)[0]
    o = oracle_mod.Oracle3D(N)
    u = np.array(t3.smooth_state(o, dims, (1.0,) * 3, seed=N))
    return o, u, dims, lambda v: o.dt(v, dims, h), lambda v, dt: o.step(v, dims, h, dt)[0]


def gpu_step(D, dims, N, u, dt, **kw):
    import torch
    ctx = (t2.make(*dims, N, **kw) if D == 2 else t3.make(dims, N, **kw))
    ud = t2.to_dev(u)
    out = torch.empty_like(ud)
    ctx.ader_step(ud, out, dt)
    torch.cuda.synchronize()
    return out.cpu().numpy().reshape(u.shape), ctx.ader_get_stats()


def worst(a, ref):
    """largest error over the variables, each by its maximum (momenta: sqrt(rho E))"""
    M = a.shape[-1]
    a, ref = a.reshape(-1, M), ref.reshape(-1, M)
    # (a face whose extrapolated trace is non-physical gives NaN on both sides)
    fine = np.isfinite(ref).all(1)
    assert np.array_equal(fine, np.isfinite(a).all(1)) and fine.any()
    a, ref = a[fine], ref[fine]
    s = np.abs(ref).max(0)
    s[1:-1] = np.maximum(s[1:-1], np.sqrt(s[0] * s[-1]))
    return float((np.abs(a - ref).max(0) / s).max())


@pytest.mark.parametrize("D,N", CASES)
@pytest.mark.parametrize("rho,vel", [(1.2, 340.0), (1e-6, 3e4), (1e12, 1.0)])
def test_units(cuda, oracle_mod, D, N, rho, vel):
    o, u, dims, dt_of, step = setup(oracle_mod, D, N)
    u[..., 0] *= rho
    u[..., 1:-1] *= rho * vel
    u[..., -1] *= rho * vel * vel
    dt = dt_of(u)
    o.base.set(fixed_iter=N + 2)
    got, _ = gpu_step(D, dims, N, u, dt, picard_fixed_iter=N + 2)
    assert worst(got, step(u, dt)) < 1e-12


@pytest.mark.parametrize("D,N", CASES)
@pytest.mark.parametrize("factor", [1e-3, 1e-9])
def test_small_time_steps(cuda, oracle_mod, D, N, factor):
    o, u, dims, dt_of, step = setup(oracle_mod, D, N)
    dt = factor * dt_of(u)
    got, st = gpu_step(D, dims, N, u, dt)
    assert worst(got, step(u, dt)) < 1e-12
    assert st["cells"] == int(np.prod(dims))


@pytest.mark.parametrize("D,N", CASES)
@pytest.mark.parametrize("kind", ["uneven", "jump", "nan"])
def test_uneven_and_redone_cells(cuda, oracle_mod, D, N, kind):
    o, u, dims, dt_of, step = setup(oracle_mod, D, N)
    nc, n = int(np.prod(dims)), N + 1
    v = u.reshape(nc, n ** D, D + 2).copy()
    if kind == "uneven":  # cells of one block from 1 to 1e4 times lighter and colder
        g = np.random.default_rng(N)
        a, b = (1e4 ** g.uniform(-1, 0, nc) for _ in range(2))
        v[..., 0] *= a[:, None]
        v[..., 1:-1] *= np.sqrt(a * b)[:, None, None]
        v[..., -1] *= b[:, None]
    elif kind == "jump":  # density down to 1/64 inside two cells
        for c in (1, nc - 1):
            low = np.arange(n ** D) % 2 == 1
            e = 0.5 * (v[c, :, 1:-1] ** 2).sum(-1) / v[c, :, 0]
            v[c, low, :-1] /= 64.0
            v[c, low, -1] -= e[low] * (1 - 1 / 64.0)
    else:
        v[nc // 2, 0, 0] = np.nan
    v = v.reshape(u.shape)
    dt = 0.1 * dt_of(v) if kind == "uneven" else 0.02 * dt_of(u)
    o.base.set(fixed_iter=3)
    got, st = gpu_step(D, dims, N, v, dt, picard_fixed_iter=3)
    assert st["cells"] == nc
    if kind != "nan":
        assert worst(got, step(v, dt)) < 1e-12
        return
    # the cell and its face neighbours are lost, every other one is what it is without it
    clean, _ = gpu_step(D, dims, N, u, dt, picard_fixed_iter=3)
    bad = ~np.isfinite(got.reshape(nc, -1)).all(1)
    assert bad[nc // 2] and bad.sum() <= 2 * D + 1
    assert np.array_equal(got.reshape(nc, -1)[~bad], clean.reshape(nc, -1)[~bad])
