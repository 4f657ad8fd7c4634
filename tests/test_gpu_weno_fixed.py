"""The fixed-point WENO reconstruction (weno_fix in csrc/ader_kernels.cuh) where it can go
wrong: stencils whose values differ by about the factor that hands them to the FP64 form,
zero momenta and sign changes, units far from one and outside the form's range, fronts
(FP64 weights) and meshes as small as the stencil.  Bar: 1e-12 of the largest value of each
stencil, per variable (a reconstruction is a sum of products of that size)."""
import numpy as np
import pytest

import workloads as W
from test_gpu_dg import to_dev

pytestmark = pytest.mark.gpu


def check(cuda, oracle_mod, N, v):
    import torch
    from paper_2409_12483_gb300 import Context
    nc = v.shape[0]
    ref = oracle_mod.Oracle(N).weno_reconstruct(np.ascontiguousarray(v)).reshape(nc, N + 1, 3)
    w = torch.empty(nc * (N + 1) * 3, dtype=torch.float64, device=cuda)
    Context(nc, N, "fv").ader_weno_reconstruct(to_dev(v, cuda), w)
    torch.cuda.synchronize()
    got = w.cpu().numpy().reshape(nc, N + 1, 3)
    scale = np.max([np.roll(np.abs(v), s, axis=0) for s in range(-N, N + 1)], axis=0)[:, None, :]
    err = np.abs(got - ref)
    assert (err <= 1e-12 * scale).all(), (err / np.maximum(scale, 1e-300)).max()


def smooth(nc, amp=0.2):
    x = (np.arange(nc) + 0.5) / nc
    return W.conserved(1 + amp * np.sin(2 * np.pi * x), 0.5 + amp * np.cos(2 * np.pi * x),
                       1 + amp * np.sin(4 * np.pi * x))


@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("ratio", [1.0 + 1e-9, 1.01, 2.0, 3.9, 4.1, 7.9, 8.1, 100.0])
def test_value_ratios(cuda, oracle_mod, N, ratio):
    v = smooth(64)
    v[20:31] *= ratio
    v[40:41] /= ratio
    check(cuda, oracle_mod, N, v)


@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("kind", ["rest", "sign", "noise", "uniform", "powers"])
def test_states(cuda, oracle_mod, N, kind):
    nc = 97
    v = smooth(nc)
    g = np.random.default_rng(N)
    if kind == "rest":
        v[:, 1] = 0.0
    elif kind == "sign":
        v[:, 1] -= v[:, 1].mean()
    elif kind == "noise":
        v *= 1 + 1e-15 * g.uniform(-1, 1, v.shape)
        v[:, 1] = 1e-17 * g.uniform(-1, 1, nc)
    elif kind == "uniform":
        v[:] = [1.0, -0.5, 2.0]
    else:  # carries at powers of two
        v[:] = np.array([1.0, 0.25, 2.0]) * (1 - 2.0 ** -53 * g.integers(0, 3, v.shape))
    check(cuda, oracle_mod, N, v)


@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("unit", [2.0 ** -40, 2.0 ** -31, 1e-6, 1e6, 2.0 ** 29, 2.0 ** 40])
@pytest.mark.parametrize("nc", [1, 3, 9, 129])
def test_units_and_meshes(cuda, oracle_mod, N, unit, nc):
    check(cuda, oracle_mod, N, smooth(nc, 0.05) * unit)
