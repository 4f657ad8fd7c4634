"""The fixed-point arithmetic of the library (csrc/ader_fix.h) and the Rusanov flux built on
it (csrc/ader_fixr.cuh), compiled for the host and measured against quadruple precision
beside the same flux in FP64: from gas nearly at rest to Mach 3000, faces without a jump to
jumps of 1e-2, along the face's normal and across it.

Bar: the largest error over the variables, each in its own size times the wave speed, is at
most twice the FP64 flux's on the same faces; the wave speed handed out for further
variables' fluxes is within the bound handed out with it."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2409_12483_gb300", "csrc")
MACHS = [1e-7, 0.1, 1.0, 3.0, 10.0, 30.0, 100.0, 300.0, 1000.0, 3000.0]


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("host") / "fixed_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-w", "-o", exe,
                    os.path.join(ROOT, "tests", "host_src", "fixed_check.cpp"),
                    os.path.join(CSRC, "ader_ops.cpp")], check=True, timeout=300)

    def run(*args):
        out = subprocess.run([exe, *map(str, args)], check=True, capture_output=True, text=True,
                             timeout=300).stdout
        return {k: float(v) for k, v in (kv.split("=") for kv in out.split())}
    return run


@pytest.mark.parametrize("D,slant", [(1, 0), (2, 0), (2, 1), (3, 0), (3, 1)])
@pytest.mark.parametrize("gamma", [1.125, 1.2, 1.4, 5.0 / 3.0, 2.0])
@pytest.mark.parametrize("jump", [1e-14, 1e-12, 1e-9, 1e-6, 1e-3, 1e-2])
def test_rusanov_flux(check, D, slant, gamma, jump):
    for mach in MACHS:
        r = check("flux", D, gamma, mach, jump, slant)
        assert r["fixed"] <= 2 * r["fp64"], (mach, r)
        assert r["over"] <= 1.0, (mach, r)
        # a fast flow along the face, and most jumps of 1e-2, are the FP64 form's
        assert slant or mach > 300 or jump > 1e-3 or r["taken"] > 4000, (mach, r)


@pytest.mark.parametrize("jump", [0.0, 1e-14, 1e-9])
def test_speed_for_further_variables(check, jump):
    """refined whatever the Euler jumps are: within 2^-49 + 2^-53 / (c s) of the units (c above
    2^-12.5, s above 3/16), which is 2^-38 at the most and 2^-46 below Mach 3 (c above 2^-5)"""
    for mach in MACHS:
        r = check("flux", 1, 1.4, mach, jump, 0)
        assert r["rel"] <= (2.0 ** -46 if mach <= 3 else 2.0 ** -38), (mach, r)


def test_small_gamma_is_left_to_fp64(check):
    assert check("flux", 1, 1.05, 1.0, 1e-6, 0)["taken"] == 0


@pytest.mark.parametrize("gamma", [1.2, 1.4, 5.0 / 3.0, 2.0])
def test_predictor_flux(check, gamma):
    for mach in MACHS:
        r = check("predictor_flux", gamma, mach)
        assert r["taken"] > 4000 and r["fixed"] <= 2 * r["fp64"], (mach, r)


def test_magnitude_of_a_change(check):
    """what the convergence tests compare: every size and either sign, within the float roundings
    of the two words and of their sum"""
    assert check("magnitude")["worst"] <= 2.0 ** -23
