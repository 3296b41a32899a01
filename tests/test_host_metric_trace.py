"""Delta^k_km of the point code (csrc/bssn_point.cuh, delta_trace), compiled for the host, against
1/2 gammabar^ab e_m h_ab in rational arithmetic from the same gammabar^ab and e_m h_ab.

A chain of six products: each of its six roundings is at most 2^-53 of the terms' magnitudes summed, and the halving is
exact.  The trace of Delta^k_ij is the same quantity, but its terms hold the rotation of h (the 1/r and cot/r
terms), which only cancels in the sum: it misses this bound on stretched metrics and near the axis.
"""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
dp = ctypes.POINTER(ctypes.c_double)
PAIRS = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


def _p(a):
    return a.ctypes.data_as(dp)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    so = str(tmp_path_factory.mktemp("metric") / "metric.so")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-Wno-unknown-pragmas",
                        os.path.join(HERE, "host_point", "metric_point.cpp"), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


@pytest.mark.parametrize("a", [1.0, 1e3])
@pytest.mark.parametrize("ratio", [1.5, 4.0, 11.0, 31.0, 101.0])
@pytest.mark.parametrize("cyl,ax", [(1, 1), (1, -1), (0, 2), (0, -1)])
@pytest.mark.parametrize("order", [4, 8])
def test_trace_of_delta(lib, order, cyl, ax, ratio, a):
    rng = np.random.default_rng(7)
    for _ in range(20):
        q = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        ev = np.array([ratio, 1.0, 1.0 / ratio]) ** 0.5      # eigenvalue ratio `ratio`, determinant 1
        g = q @ np.diag(ev) @ q.T
        x = np.linspace(-0.05, 0.05, 11)
        y = np.zeros((24, 11, 11, 11))
        for s, (i, j) in enumerate(PAIRS):
            k, ph = rng.uniform(0.5, 2.0, 3), rng.uniform(0, 6, 3)
            wave = np.sin(k[0] * x + ph[0])[None, None, :] + np.sin(k[1] * x + ph[1])[None, :, None] + \
                np.sin(k[2] * x + ph[2])[:, None, None]
            y[s] = g[i, j] - (i == j) + 0.02 * ev.min() * wave
        y[12] = 1.0
        geo = np.array([100.0 / (12 if order == 4 else 840)] * 3 + [a, 0.0 if cyl else a, 0.0 if cyl else 0.7 * a])
        gi, dh, dtr = np.empty(6), np.empty(18), np.empty(3)
        lib.metric_point(cyl, ax, order, _p(y), _p(geo), _p(gi), _p(dh), _p(dtr))
        for m in range(3):
            terms = [(1 if i == j else 2) * Fr(float(gi[s])) * Fr(float(dh[6 * m + s])) for s, (i, j) in enumerate(PAIRS)]
            bound = 6 * sum(abs(t) for t in terms) / 2 ** 54 * (1 + Fr(1, 2 ** 40))
            assert abs(Fr(float(dtr[m])) - sum(terms) / 2) <= bound
