"""The step-size factor 0.9 (tol / err)^(1/3) of the FP64 group-per-ray
integrator (step_factor.h), compiled for the host."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1404_3363_gb300", "csrc")


@pytest.fixture(scope="module")
def factor(tmp_path_factory):
    d = tmp_path_factory.mktemp("step_factor")
    src = d / "f.cpp"
    src.write_text('#include "step_factor.h"\n'
                   'extern "C" double f(double tol, double err) { return ivv::coop_step_factor(tol, err); }\n')
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(d / "f.so")],
                   check=True)
    f = ctypes.CDLL(str(d / "f.so")).f
    f.argtypes, f.restype = [ctypes.c_double] * 2, ctypes.c_double
    return f


@pytest.mark.parametrize("tol", [1e-10, 1e-5, 1e-2])
@pytest.mark.parametrize("err", [math.inf, 1.7e308, 1e300, 3.5e38, 3.3e38, 1e37, 1e36, 1e-36, 1e-38, 1e-45, 1e-300])
def test_errors_beyond_single_precision(factor, tol, err):
    """Infinite (a slope at a point with det J = 0), huge and tiny errors: a
    number, so that the step shrinks or grows by the limits of the control."""
    want = 0.9 * float(np.cbrt(tol / err))
    assert factor(tol, err) == pytest.approx(want, rel=1e-12)


def test_double_precision(factor):
    """Less than a rounding of the root (the Newton step's) and one of the
    product: within two units in the last place, over the whole range that takes
    the FP32 start."""
    rng = np.random.default_rng(7)
    third = np.longdouble(1) / 3
    for _ in range(20000):
        tol, err = 10.0 ** rng.uniform(-24, 12, 2)
        want = np.longdouble(0.9) * (np.longdouble(tol) / np.longdouble(err)) ** third
        assert abs(np.longdouble(factor(tol, err)) / want - 1) <= 4.5e-16
