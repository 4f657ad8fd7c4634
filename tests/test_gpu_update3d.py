"""lambda_max of the 3D update kernel (csrc/ader_kernels3d.cuh): blocks that the FP32
screen ends and blocks that go on to FP64, in uniform flow (every subcell ties), with one
fast cell among quiet ones, in smooth flow and in units far from one; meshes with a partial
last block.  Bar: the time steps, and so the end time, are the oracle's to 1e-13."""
import numpy as np
import pytest

import test_gpu_3d as t3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 7])
@pytest.mark.parametrize("kind", ["uniform", "fast cell", "smooth", "units"])
@pytest.mark.parametrize("dims", [(3, 2, 5), (1, 1, 1), (4, 4, 3)])
def test_time_steps(cuda, oracle_mod, N, kind, dims):
    import torch
    if N == 7 and dims == (4, 4, 3):
        pytest.skip("the oracle takes long")
    o = oracle_mod.Oracle3D(N)
    u = np.array(t3.smooth_state(o, dims, (1.0,) * 3, seed=N))
    nc = int(np.prod(dims))
    v = u.reshape(nc, (N + 1) ** 3, 5).copy()
    if kind in ("uniform", "fast cell"):
        v[:] = [1.0, 0.3, -0.2, 0.1, 2.57]
    if kind == "fast cell":
        v[nc // 2] = [1.0, 0.31, -0.2, 0.1, 2.6]
    if kind == "units":
        v *= np.array([1e-6, 3e-2, 3e-2, 3e-2, 9e2])
    v = v.reshape(u.shape)
    h = tuple(1.0 / d for d in dims)
    ctx = t3.make(dims, N)
    ud = t3.to_dev(v)
    assert abs(ctx.ader_compute_dt(ud, 0.0, -1.0) / o.dt(v, dims, h) - 1) < 1e-13
    steps, t, _ = ctx.ader_solve(ud, max_steps=2)
    torch.cuda.synchronize()
    dt1 = o.dt(v, dims, h)
    dt2 = o.dt(np.array(o.step(v, dims, h, dt1)[0]), dims, h)
    assert steps == 2 and abs(t / (dt1 + dt2) - 1) < 1e-13
