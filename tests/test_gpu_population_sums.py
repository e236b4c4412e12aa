"""FP64 sums over the populations of FP32 nodes (lbm::node_sums_fp64): where
the integer path takes a node, each sum is the exact one rounded once, so it
equals math.fsum of the terms; a node with denormals, infinities, NaN or a gap
of more than 30 binades is left to the FP64 additions, each of which rounds
to 2^-53 of a partial sum (of at most nine terms of the largest size)."""
import ctypes as C
import math
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
pytestmark = pytest.mark.gpu
ROWS = (np.array([1] * 9), np.array([0, 1, 0, -1, 0, 1, -1, -1, 1]), np.array([0, 0, 1, 0, -1, 1, 1, -1, -1]))


def nodes():
    """(n, 18) float32 and what the integer path should do with each node
    (True, False, or None where the draw decides)."""
    r = np.random.default_rng(11)
    out, want = [], []

    def add(v, exact=None):
        out.append(np.asarray(v, dtype=np.float32).reshape(18))
        want.append(exact)

    for _ in range(2000):
        add(r.uniform(-0.5, 0.5, 18) * 2.0 ** -r.integers(0, 12, 18), True)
        add(np.ldexp(r.uniform(0.5, 1, 18) * r.choice([-1, 1], 18), -r.integers(0, 40, 18)))
        v = r.uniform(-1, 1, 18)                                       # pairs that cancel
        v[5:9] = -v[1:5]
        v[14:18] = -v[10:14]
        add(v, None)
        add(r.uniform(-1, 1, 18) * (r.random(18) < 0.4))               # zeros among values
    add(np.zeros(18), True)
    add(-np.zeros(18), True)
    for gap, exact in ((29, True), (30, True), (31, False), (60, False)):
        for s in (1.0, -1.0):
            for base in (1.0, 2.0 ** 90, 2.0 ** -60):
                v = np.full(18, base, dtype=np.float64)
                v[[3, 12]] = s * base * 2.0 ** -gap
                add(v, exact)
    for big in (2.0 ** 127, -2.0 ** 127, float(np.finfo(np.float32).max)):
        add(np.full(18, big), True)                                    # beyond FP32, not beyond FP64
    # ties of the one rounding: 2^23 + 1 units and halves 30 binades below it
    for lo in (1.0, -1.0, 3.0, 1.5):
        v = np.zeros(18)
        v[0], v[1], v[9], v[10] = 2.0 ** 24 - 1, lo * 2.0 ** -6, 2.0 ** 24 - 1, lo * 2.0 ** -6
        add(v, True)
    for bad in (2.0 ** -140, -2.0 ** -149, np.inf, -np.inf, np.nan):
        for k in (0, 8, 9, 17):
            v = np.full(18, 0.25)
            v[k] = bad
            add(v, False)
    add(np.full(18, 2.0 ** -135), False)
    add(np.full(18, 2.0 ** -126), True)                                # smallest normal number
    return np.stack(out), want


def test_sums_are_exact_and_rounded_once(tmp_path):
    from paper_1809_08683_gb300 import lbm
    so = str(tmp_path / "sums_check.so")
    subprocess.check_call([lbm._nvcc(), *lbm.NVCC_FLAGS, "-o", so, os.path.join(HERE, "sums_check.cu")])
    v, want = nodes()
    out, exact = np.empty((len(v), 4)), np.empty(len(v), dtype=np.int32)
    ptr = lambda a, t: a.ctypes.data_as(C.POINTER(t))  # noqa: E731
    assert C.CDLL(so).sums_check(ptr(v, C.c_float), ptr(out, C.c_double), ptr(exact, C.c_int), C.c_int(len(v))) == 0
    w = v.astype(np.float64)
    for i in range(len(v)):
        assert want[i] is None or bool(exact[i]) == want[i], (i, v[i])
        for k, (half, row) in enumerate(((0, 0), (0, 1), (0, 2), (9, 0))):
            used = ROWS[row] != 0
            terms = w[i, half:half + 9][used] * ROWS[row][used]
            got = out[i, k]
            if not np.isfinite(terms).all():
                ref = terms.sum()
                assert (math.isnan(got) and math.isnan(ref)) or got == ref, (i, k)
            elif exact[i]:
                assert got == math.fsum(terms), (i, k, v[i])
            else:
                assert abs(got - math.fsum(terms)) <= 9 * 9 * 2.0 ** -53 * np.abs(terms).max(), (i, k)
    assert 0.3 < exact.mean() < 1
