"""The time loop's lambda_max on the systems whose interface kernels carry more than
the Euler variables: every step of a solve takes the time step that ader_compute_dt
(another kernel) finds for the state it starts from, and a solve repeats itself bit for
bit.  Smooth fine meshes: the speeds of a tile lie closer than FP32 resolves, so the
interface kernel's float-float screen decides."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("system", ["reacting", "tracer"])
@pytest.mark.parametrize("N,nc", [(3, 30011), (5, 20000)])
def test_loop_time_steps(cuda, system, N, nc):
    import torch
    from paper_2409_12483_gb300 import Context
    ctx = Context(nc, N, "dg", system=system)
    x = torch.tensor(ctx.node_coords(), device="cuda")
    w = 2 * np.pi * x
    rho, p = 1 + 0.1 * torch.sin(w + 0.3), 1 + 0.05 * torch.cos(2 * w)
    E = p / 0.4 + 0.5 * rho * 0.25
    extra = [rho * 0.5, rho * 0.2 * torch.cos(w)] if system == "reacting" else [1 + 0.1 * torch.sin(3 * w)]
    u0 = torch.stack([rho, 0.5 * rho, E, *extra], -1).reshape(-1).contiguous()
    times = set()
    for _ in range(3):
        u = u0.clone()
        _, t, _ = ctx.ader_solve(u, max_steps=5)
        times.add((t, u.sum().item()))
    assert len(times) == 1
    u, v, t = u0.clone(), torch.empty_like(u0), 0.0
    for _ in range(5):
        dt = ctx.ader_compute_dt(u)
        ctx.ader_step(u, v, dt)
        u, v = v, u
        t += dt
    assert abs(times.pop()[0] - t) < 1e-14 * t
