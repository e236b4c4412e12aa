"""Relative accuracy of s_q and sigma_e in FP32 at small viscosity.

Both rates vanish with the viscosity, and the changes of the moments that
they relax are proportional to them.  From the viscosity on, each result
below takes at most 12 roundings (constants among them) and no difference of
nearly equal numbers, so it is within 12 * 2^-24 of itself."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("node_rates") / "node_rates.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                           os.path.join(HERE, "node_rates.cpp"), "-o", so])
    return C.CDLL(so)


@pytest.mark.parametrize("mu0", [2e-5, 1.7e-4, 1e-3, 0.03, 0.1, 0.5])
@pytest.mark.parametrize("mu_j", [0.7, 2.8, 6.1])
def test_vanishing_rates_keep_relative_accuracy(helper, mu0, mu_j):
    a, b = np.empty(2), np.empty(2)
    ptr = lambda v: v.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
    helper.node_rates(C.c_double(mu0), C.c_double(mu_j), ptr(a), ptr(b))
    assert np.all(b != 0) and np.all(np.abs(a - b) <= 12 * 2.0 ** -24 * np.abs(b)), (a / b - 1)
