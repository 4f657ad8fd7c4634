"""The limiter's correction of an untroubled cell next to a troubled one: what it takes off
is the flux that the interface kernel put on, whatever form that flux has, so a step
conserves mass, momentum and energy at any Mach number.  Uniform velocity, small random
jumps at every face (the fixed-point flux's range) and a strict maximum principle, so that
about half of the cells are troubled.

Bar: 2e-14 of the totals, as the limiter's other conservation test: a step's own rounding is a
few 2^-53 of each cell's values."""
import numpy as np
import pytest

from test_gpu_dg import to_dev
from test_gpu_limiter import make
from test_oracle_limiter import conserved

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 3, 5, 7])
@pytest.mark.parametrize("mach", [0.1, 3.0, 100.0, 1000.0])
@pytest.mark.parametrize("bc", ["periodic", "outflow"])
def test_step_is_conservative(cuda, oracle_mod, N, mach, bc):
    import torch
    nc = 64
    o = oracle_mod.Oracle(N)
    g = np.random.default_rng(N)
    cell = lambda a: 1 + a * g.uniform(-1, 1, (nc, 1))
    rho = cell(1e-3) * (1 + 2e-4 * g.uniform(-1, 1, (nc, N + 1)))
    u = conserved(rho, mach * np.sqrt(1.4) * np.ones(rho.shape), cell(1e-4) * np.ones(rho.shape))
    if bc == "outflow":  # the ends uniform, so that what leaves and enters is the same
        u[:4] = u[-4:] = conserved(np.ones(4), mach * np.sqrt(1.4) * np.ones(4), np.ones(4))[0]
    dt = o.dg_dt(u, 1.0 / nc)
    ctx = make(nc, N, bc=bc, limiter=1, nad_delta0=0.0, nad_eps=0.0)
    ud = to_dev(u, cuda)
    out = torch.empty_like(ud)
    ctx.ader_step(ud, out, dt)
    flags = ctx.ader_get_troubled().cpu().numpy()
    torch.cuda.synchronize()
    assert np.count_nonzero(flags[1:] != flags[:-1]) >= 8
    w = o.table("w")[:N + 1]
    tot = lambda U: np.einsum("ckr,k->r", U.reshape(nc, N + 1, 3), w) / nc
    np.testing.assert_allclose(tot(out.cpu().numpy()), tot(u), rtol=2e-14)
