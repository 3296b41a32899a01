"""The bodies that the kernels run per point (csrc/nr_stage.cuh), compiled for the host, against the oracle.

The difference sums come from where the kernels take them: the stored first differences of both pipes, the
tables of raw sums in local and in shared memory (in the latter filled by four warps in turn, the last tile
with idle lanes), the constraints' tables.  Tables start as NaN, so an entry that is read but not filled shows.
Tolerances as for the inline formulation: 1e-12 of the largest component of each tensor, of the largest
Hamiltonian constraint, and of the largest momentum component.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2505_00097_gb300 import workloads as W
from tests._common import assert_close

HERE = os.path.dirname(os.path.abspath(__file__))
RHS, SPREAD, HAM, MOM = 0, 1, 2, 3


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    so = str(tmp_path_factory.mktemp("stage") / "stage.so")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-Wno-unknown-pragmas",
                        "-I", os.path.join(HERE, "host_point", "stub"), os.path.join(HERE, "host_point", "stage_point.cpp"),
                        "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(so)
    dp = ctypes.POINTER(ctypes.c_double)
    L.stage_point.argtypes = [ctypes.c_int, ctypes.POINTER(ctypes.c_int), dp, dp, dp, ctypes.c_double, dp, dp,
                              ctypes.c_int, ctypes.c_int]
    L.stage_point.restype = None
    return L


def _run(L, spec, y, which, out_len):
    dp = ctypes.POINTER(ctypes.c_double)
    ko = spec.get("ko_sigma", 0.3)
    sig = (ctypes.c_double * 24)(*(list(ko) if isinstance(ko, (list, tuple)) else [ko] * 24))
    out = np.zeros(out_len)
    L.stage_point(int(spec["coords"]), (ctypes.c_int * 3)(*spec["N"]), (ctypes.c_double * 3)(*spec["ampl"]),
                  (ctypes.c_double * 3)(*spec["sinhw"]), sig, float(spec.get("eta", 2.0)), y.ctypes.data_as(dp),
                  out.ctypes.data_as(dp), which, int(spec["NG"]))
    return out


def _order8(spec):
    return dict(spec, NG=5, ko_sigma=[0.3] * 17 + [0.99] * 7)


CYL = dict(rho_max=5.0, z_max=5.0)
GRIDS = [
    ("sinhsph_general", W.sinh_spherical((9, 7, 6))),
    ("sinhcyl_general", W.sinh_cylindrical((9, 4, 11), **CYL)),
    ("spherical_general", W.spherical((8, 6, 8))),
    ("sinhsph_two_point_phi", W.sinh_spherical((11, 9, 2))),
    ("sinhcyl_two_point_phi", W.sinh_cylindrical((11, 2, 13), **CYL)),
    ("sinhsph_general_ord8", _order8(W.sinh_spherical((11, 10, 6)))),
    ("sinhcyl_general_ord8", _order8(W.sinh_cylindrical((11, 6, 13), **CYL))),
    ("sinhsph_two_point_phi_ord8", _order8(W.sinh_spherical((13, 11, 2)))),
    ("sinhcyl_two_point_phi_ord8", _order8(W.sinh_cylindrical((13, 2, 15), **CYL))),
]
IDS = [g[0] for g in GRIDS]


def _state(spec, seed, smooth):
    o = Oracle(spec)
    y = W.random_state(o.n, seed=seed, smooth=smooth)
    o.inner_bc(y)
    return o, y


@pytest.mark.parametrize("smooth", [True, False], ids=["smooth", "noise"])
@pytest.mark.parametrize("name,spec", GRIDS, ids=IDS)
def test_rhs_bodies_match_the_oracle(lib, name, spec, smooth):
    o, y = _state(spec, 21, smooth)
    ref = o.rhs(y)
    m = o.interior_mask()
    got = _run(lib, spec, y, RHS, y.size)
    assert_close(got, ref, o.T, 1e-12, mask=m, what=f"{name} k_rhs body")
    spread = _run(lib, spec, y, SPREAD, y.size)
    assert np.array_equal(got, spread)            # the same sums from the other table


@pytest.mark.parametrize("name,spec", GRIDS, ids=IDS)
def test_constraint_bodies_match_the_oracle(lib, name, spec):
    o, y = _state(spec, 22, True)
    m = o.interior_mask()
    ref = o.hamiltonian(y)[0]
    got = _run(lib, spec, y, HAM, o.T)
    assert np.abs(got[m] - ref[m]).max() <= 1e-12 * np.abs(ref[m]).max()
    ref = o.momentum(y)[0]
    got = _run(lib, spec, y, MOM, 3 * o.T).reshape(3, o.T)
    assert np.abs(got[:, m] - ref[:, m]).max() <= 1e-12 * np.abs(ref[:, m]).max()
    # the table divided among four warps holds the same sums
    assert np.array_equal(_run(lib, spec, y, HAM + 2, o.T), _run(lib, spec, y, HAM, o.T))
    assert np.array_equal(_run(lib, spec, y, MOM + 2, 3 * o.T).reshape(3, o.T), got)


SPH, CYL = 0, 1


@pytest.mark.parametrize("tiles,outer,order,two,shape", [
    (1, 1, 4, 1, 0), (440, 16, 4, 1, 0), (441, 16, 4, 1, 1), (592, 16, 4, 1, 1), (593, 16, 4, 1, 2), (608, 0, 4, 0, 1),
    (608, 1, 4, 0, 2), (609, 1, 4, 0, 0), (896, 16, 4, 1, 0), (897, 16, 4, 1, 2), (1216, 200, 4, 0, 2), (1217, 16, 4, 0, 3),
    (1824, 0, 4, 0, 3), (1824, 1, 4, 0, 2), (1825, 30, 4, 0, 3), (8192, 50, 4, 1, 3),
    (288, 16, 8, 1, 0), (440, 16, 8, 1, 0), (441, 16, 8, 1, 2), (441, 16, 8, 0, 1), (700, 16, 8, 1, 0), (1100, 29, 8, 0, 2), (1101, 29, 8, 0, 3),
    (1824, 1, 8, 0, 3),
])
def test_launch_shape_lines(lib, tiles, outer, order, two, shape):
    """The rule at its lines, on 152 SMs and on twice as many with twice the work."""
    lib.stage_shape.argtypes = [ctypes.c_int] * 4 + [ctypes.c_long] * 2
    assert lib.stage_shape(SPH, order, two, 152, tiles, outer) == shape
    if tiles % 4 == 0:
        assert lib.stage_shape(SPH, order, two, 304, 2 * tiles, 2 * outer) == shape
    # cylindrical coordinates differ with a two-point azimuth and 8th order: one round of two spread blocks
    if order == 8 and two and 304 < tiles + outer <= 456:
        shape = 2
    assert lib.stage_shape(CYL, order, two, 152, tiles, outer) == shape
