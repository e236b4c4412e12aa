"""FP64 square root of the per-node arithmetic (lbm::root, lbm_node.cuh).

With t = x y (1 + d), |d| <= 2^-53, the third-order step removes the error of
y and half of d, so the result is within 1/4 + 1/2 ulp of the root plus the
series' remainder (5/16) e^3 < 2^-57: at most one ulp from the correctly
rounded root."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1809_08683_gb300 import lbm

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.gpu
def test_root_within_one_ulp(tmp_path):
    so = str(tmp_path / "root_check.so")
    subprocess.check_call([lbm._nvcc(), *lbm.NVCC_FLAGS, "-o", so, os.path.join(HERE, "root_check.cu")])
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.uniform(0.05, 8.0, 100_000), np.exp(rng.uniform(-40, 40, 50_000)),
                        1.0 + np.arange(-500, 500) * 2.0 ** -52, [0.0, -1.0, 1.0, 4.0, 0.25]])
    a, b = np.empty_like(x), np.empty_like(x)
    ptr = lambda v: v.ctypes.data_as(C.POINTER(C.c_double))  # noqa: E731
    assert C.CDLL(so).root_check(ptr(x), ptr(a), ptr(b), C.c_int(x.size)) == 0
    ok = x >= 0
    assert np.all(np.abs(a[ok] - b[ok]) <= np.spacing(b[ok])) and a[x == 0.0][0] == 0.0
    assert np.isnan(a[x < 0]).all()
