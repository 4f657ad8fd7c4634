"""The further variables of the reacting and tracer systems, each measured by its own size:
species and tracers far smaller or larger than the Euler variables, a species that only its
source brings up from zero, reaction frequencies, small time steps.

Both sides run a fixed number of outer iterations, and the tolerance is far below what
either can reach, so that the inner iterations end at their cap and no early stop is in the
comparison.  Bar: 1e-12 of each variable's largest value (momentum: sqrt(rho E)); the two
species are one oscillator, c2 enters c1 as dt c2 and c1 enters c2 as dt omega^2 c1."""
import numpy as np
import pytest

import test_gpu_fixed_systems as fs

pytestmark = pytest.mark.gpu


def errors(got, ref):
    M = ref.shape[-1]
    got, ref = got.reshape(-1, M), ref.reshape(-1, M)
    s = np.abs(ref).max(0)
    s[1] = max(s[1], np.sqrt(s[0] * s[2]))
    return np.abs(got - ref).max(0) / np.maximum(s, 1e-300)


def run_reacting(oracle_mod, N, u, omega, factor, iters=6):
    nc = len(u)
    o = oracle_mod.ReactingOracle(N, omega=omega, fixed_iter=iters, tol=1e-25)
    dt = factor * o.dg_dt(u, 1.0 / nc)
    got, _ = fs.gpu_step(u, N, dt, "reacting", omega=omega, picard_fixed_iter=iters,
                         picard_tol=1e-25)
    return errors(got, o.dg_step(u, 1.0 / nc, dt)[0])


@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("c1,c2", [(1e-4, 3.0), (1e3, 1e-2), (1.0, 1.0), (1.0, 1e-9), (1e-9, 1e-9),
                                   (1e8, 1e8)])
@pytest.mark.parametrize("omega", [0.0, 2.0, 30.0])
def test_species(cuda, oracle_mod, N, c1, c2, omega):
    o = oracle_mod.ReactingOracle(N, omega=omega)
    e = run_reacting(oracle_mod, N, fs.reacting(o, 33, 3, c1, c2), omega, 1.0)
    assert e.max() < 1e-12


@pytest.mark.parametrize("N", [1, 4, 7])
@pytest.mark.parametrize("which", [3, 4])
@pytest.mark.parametrize("size", [1.0, 1e-6, 1e6])
@pytest.mark.parametrize("factor", [1.0, 1e-3, 1e-6])
def test_species_from_zero(cuda, oracle_mod, N, which, size, factor):
    """an oscillator at its turning point: one species is zero everywhere"""
    o = oracle_mod.ReactingOracle(N, omega=2.0)
    u = fs.reacting(o, 33, 3, size, size)
    u[..., which] = 0.0
    e = run_reacting(oracle_mod, N, u, 2.0, factor)
    assert e.max() < 1e-12


@pytest.mark.parametrize("N", [1, 3, 6])
@pytest.mark.parametrize("a", [1e-9, 1e-6, 1.0, 1e5, 1e9])
@pytest.mark.parametrize("factor", [1.0, 1e-6])
def test_tracer(cuda, oracle_mod, N, a, factor):
    nc, iters = 33, 6
    o = oracle_mod.NCOracle(N, tol=1e-25, fixed_iter=iters)
    u = fs.tracer(o, nc, 2, a)
    dt = factor * o.dt(u, 1.0 / nc)
    got, _ = fs.gpu_step(u, N, dt, "tracer", picard_fixed_iter=iters, picard_tol=1e-25)
    assert errors(got, o.step(u, 1.0 / nc, dt)[0]).max() < 1e-12
