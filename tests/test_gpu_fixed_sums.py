"""The integer-pipe difference sums on the device against the host build of the same header, bit for bit: the
device takes other instructions for the shift, the high product and the leading zeros.  The host build is
checked against rational arithmetic in test_host_fixed_sums.py and test_host_fixed_edges.py.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2505_00097_gb300 import build as BUILD  # noqa: E402
from tests.test_host_fixed_edges import D1, KC, TOPS, edge_rows  # noqa: E402
from tests.test_host_fixed_sums import _rows  # noqa: E402

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
dp = ctypes.POINTER(ctypes.c_double)


def _p(a):
    return a.ctypes.data_as(dp)


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if shutil.which("g++") is None:
        pytest.skip("g++ not found")
    tmp = tmp_path_factory.mktemp("fixed_device")
    src = os.path.join(HERE, "host_point")
    host, dev = str(tmp / "host.so"), str(tmp / "device.so")
    for cmd in (["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-Wno-unknown-pragmas",
                 os.path.join(src, "fixed_point.cpp"), "-o", host],
                [BUILD.nvcc(), *BUILD.ARCH, "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "static",
                 os.path.join(src, "fixed_device.cu"), "-o", dev]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    return ctypes.CDLL(host), ctypes.CDLL(dev)


def _same(a, b):
    assert np.array_equal(np.isnan(a), np.isnan(b))
    ok = ~np.isnan(a)
    assert np.array_equal(a[ok].view(np.int64), b[ok].view(np.int64))


def _all_rows(order):
    rng = np.random.default_rng(40 + order)
    special = _rows(rng, "noise", 60, 9)
    special[np.arange(60), rng.integers(0, 9, 60)] = rng.choice([np.inf, -np.inf, np.nan, 1e308, 1e-290, 5e-324, 0.0], 60)
    return np.ascontiguousarray(np.concatenate([edge_rows(order), _rows(rng, "smooth", 3000, 9), _rows(rng, "noise", 3000, 9),
                                                _rows(rng, "binades", 3000, 9), special]))


@pytest.mark.parametrize("order", [4, 8])
def test_first_differences(libs, order):
    host, dev = libs
    f = _all_rows(order)
    n = len(f)
    out, fp, got = np.empty(n), np.empty(n), np.empty(n)
    host.fixed_d1(order, _p(f), ctypes.c_long(n), _p(out), _p(fp))
    assert dev.device_d1(order, _p(f), ctypes.c_long(n), _p(got)) == 0
    _same(got, out)


@pytest.mark.parametrize("order", [4, 8])
def test_mixed_differences(libs, order):
    host, dev = libs
    rng = np.random.default_rng(50 + order)
    blocks = [_rows(rng, kind, 1, 81) for kind in ("smooth", "noise", "binades") for _ in range(100)]
    sgn = np.array([np.sign(D1[order].get(j - 4, 0)) for j in range(9)])
    for x in TOPS:
        blocks += [(s * x * sgn[:, None] * sgn[None, :]).reshape(1, 81) for s in (-1.0, 1.0)]
    f = np.ascontiguousarray(np.concatenate(blocks))
    n = len(f)
    out, fp, got = np.empty(n), np.empty(1), np.empty(n)
    for i in range(n):
        one = np.empty(1)
        host.fixed_mix(order, _p(f[i]), _p(one), _p(fp))
        out[i] = one[0]
    assert dev.device_mix(order, _p(f), ctypes.c_long(n), _p(got)) == 0
    _same(got, out)


def test_subtraction(libs):
    host, dev = libs
    rng = np.random.default_rng(60)
    n = 20000
    a = rng.uniform(-1, 1, n) * 2.0 ** rng.integers(-300, 300, n)
    b = a * rng.choice([1.0, 1.0 + 1e-9, 0.7, -1.0, 1.3, 0.0, 2.0 ** -53, 2.0 ** -60], n)
    a[:4], b[:4] = (0.0, np.inf, 1e300, 1.0), (0.0, 1.0, -1e300, -2.0 ** -53)
    out, got = np.empty(n), np.empty(n)
    host.fixed_sub(_p(a), _p(b), ctypes.c_long(n), _p(out))
    assert dev.device_sub(_p(a), _p(b), ctypes.c_long(n), _p(got)) == 0
    _same(got, out)


@pytest.mark.parametrize("ax", [-1, 1, 2])
@pytest.mark.parametrize("order", [4, 8])
def test_advection_and_dissipation(libs, order, ax):
    host, dev = libs
    rng = np.random.default_rng(70 + order + ax)
    n, c = 120, 5 + 11 * (5 + 11 * 5)
    y, par = np.zeros((n, 24, 1331)), np.empty((n, 4))
    out, fp, got = np.empty(n), np.empty(1), np.empty(n)
    for i in range(n):
        kind = ("smooth", "noise", "binades", "top")[i % 4]
        vet = rng.uniform(-0.3, 0.3, 3) * 10.0 ** rng.uniform(-8, 0, 3) * (rng.uniform(size=3) > 0.15)
        D, sigma = 10.0 ** rng.uniform(-3, 3, 3), float(rng.choice([0.0, 0.3, 0.99, 1e-6]))
        if kind == "top":
            x = TOPS[(i // 4) % len(TOPS)]
            f = rng.choice([-1.0, 1.0], 1331) * x
            sigma, D = 1.0, np.full(3, x / float(KC[order]))
            vet = rng.choice([-1.0, 1.0], 3) * float(KC[order])
        else:
            f = _rows(rng, kind, 1, 1331)[0]
        f = np.ascontiguousarray(f)
        y[i, 0], y[i, 17:20, c], par[i, :3], par[i, 3] = f, vet, D, sigma
        one = np.empty(1)
        host.fixed_advko(ax, order, _p(f), _p(np.ascontiguousarray(vet)), _p(np.ascontiguousarray(D)),
                         ctypes.c_double(sigma), _p(one), _p(fp))
        out[i] = one[0]
    assert dev.device_adv(ax, order, _p(y), _p(par), ctypes.c_long(n), _p(got)) == 0
    _same(got, out)
