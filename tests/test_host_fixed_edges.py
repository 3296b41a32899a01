"""The integer-pipe difference sums (csrc/fixed_sum.cuh) with values at the top of a power of two, compiled for the
host, against rational arithmetic: the largest mantissas, with signs that make every partial sum as large as it gets.

The bounds are those of the sums at any values: one rounding of the result, 2^-53 of it, plus one unit of the
alignment (2^-(52 + SH) of the largest value) per value and unit of weight; the advection + dissipation sum also
the alignment of its coefficients and what its integers drop at the end.  Values of one exponent align
exactly, so a first difference of them is the correctly rounded one.
"""
import ctypes
import itertools
import os
import shutil
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
D1 = {4: {-2: 1, -1: -8, 1: 8, 2: -1}, 8: {-4: 3, -3: -32, -2: 168, -1: -672, 1: 672, 2: -168, 3: 32, 4: -3}}
UP = {4: {-1: -3, 0: -10, 1: 18, 2: -6, 3: 1},
      8: {-3: -5, -2: 60, -1: -420, 0: -378, 1: 1050, 2: -420, 3: 140, 4: -30, 5: 3}}
KO = {4: (1, -6, 15, -20, 15, -6, 1), 8: (1, -10, 45, -120, 210, -252, 210, -120, 45, -10, 1)}
KC = {4: Fr(12, 64), 8: Fr(840, 1024)}
# 1 - 2^-53 is the last FP64 number below 1; differences of opposite signs reach 2^-32 below the next power of two
TOPS = [1 - 2.0 ** -k for k in (53, 52, 45, 40, 34, 33, 32, 31, 30, 20, 1)]
dp = ctypes.POINTER(ctypes.c_double)


def _p(a):
    return a.ctypes.data_as(dp)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    so = str(tmp_path_factory.mktemp("fixed_edges") / "fixed.so")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-Wno-unknown-pragmas",
                        os.path.join(HERE, "host_point", "fixed_point.cpp"), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def edge_rows(order):
    """Rows of 9 values: every sign pattern over the offsets, at each top value, and one exponent higher and lower."""
    M = order // 2
    offs = [o for o in range(-M, M + 1) if o]
    rows = []
    for x in TOPS:
        for signs in itertools.product((-1.0, 1.0), repeat=len(offs)):
            r = np.zeros(9)
            for o, s in zip(offs, signs):
                r[4 + o] = s * x
            rows.append(r)
    # values next to the top with different mantissas, and only one pair of them non-zero
    for o, (a, b), s in itertools.product(range(1, M + 1), itertools.product(TOPS, repeat=2), (-1.0, 1.0)):
        r = np.zeros(9)
        r[4 + o], r[4 - o] = s * a, -s * b
        rows.append(r)
    f = np.array(rows)
    return np.ascontiguousarray(np.concatenate([f, f * 2.0 ** 60, f * 2.0 ** -60]))


@pytest.mark.parametrize("order", [4, 8])
def test_first_difference_at_the_top_of_a_binade(lib, order):
    f = edge_rows(order)
    out, fp = np.empty(len(f)), np.empty(len(f))
    lib.fixed_d1(order, _p(f), ctypes.c_long(len(f)), _p(out), _p(fp))
    exact = [sum(w * Fr(float(row[4 + j])) for j, w in D1[order].items()) for row in f]
    bad = [(row.tolist(), o, float(e)) for row, o, e in zip(f, out, exact) if abs(Fr(float(o)) - e) > abs(e) / 2 ** 53]
    assert not bad, (len(bad), bad[:3])


@pytest.mark.parametrize("order", [4, 8])
def test_mixed_difference_at_the_top_of_a_binade(lib, order):
    """Sign patterns that make the row differences, or the difference of the rows, as large as they get."""
    weight = sum(abs(w) for w in D1[order].values())
    sh = 5 if order == 4 else 9
    sgn = {o: (1.0 if w > 0 else -1.0) for o, w in D1[order].items()}
    for x, flip in itertools.product(TOPS, (-1.0, 1.0)):
        for kind in ("extreme", "one sign per row", "corners"):
            f = np.zeros((9, 9))
            for i, j in itertools.product(D1[order], repeat=2):
                if kind == "extreme":
                    f[4 + i, 4 + j] = flip * sgn[i] * sgn[j] * x
                elif kind == "one sign per row":
                    f[4 + i, 4 + j] = flip * (x if i > 0 else -x) * (1.0 if j > 0 else -1.0)
                elif abs(i) == 1 and abs(j) == 1:
                    f[4 + i, 4 + j] = flip * i * j * x
            out, fp = np.empty(1), np.empty(1)
            lib.fixed_mix(order, _p(f), _p(out), _p(fp))
            rows = {i: sum(w * Fr(float(f[4 + i, 4 + j])) for j, w in D1[order].items()) for i in D1[order]}
            exact = sum(w * rows[i] for i, w in D1[order].items())
            row = max(abs(r) for r in rows.values())
            row_err = row / 2 ** 53
            bound = weight * row_err + (abs(exact) + weight * row_err) / 2 ** 53 + weight * (row + row_err) / 2 ** (52 + sh)
            assert abs(Fr(float(out[0])) - exact) <= bound, (x, flip, kind, out[0], float(exact))


@pytest.mark.parametrize("ax", [-1, 1, 2])
@pytest.mark.parametrize("order", [4, 8])
def test_advection_and_dissipation_at_the_top_of_a_binade(lib, order, ax):
    """Values, shift and scales at the largest mantissas; signs that maximise the upwind sum, the dissipation sum, and
    their cross products, for both directions of the shift."""
    G = len(KO[order]) // 2
    up, ko = sum(abs(w) for w in UP[order].values()), sum(abs(w) for w in KO[order])
    sh = 2 if order == 4 else 5
    weights = 3 * (up + ko) + (2 * (768 + 512) if order == 8 else 2 * 48)
    last = Fr(1, 2 ** 52) if order == 4 else Fr(6, 2 ** 48) + Fr(1, 2 ** 46)
    for x, follow, flip, vs, kap in itertools.product(TOPS[:8], ("up", "ko"), (-1.0, 1.0), (-1.0, 1.0), (1.0, 2.0 ** -30)):
        f = np.zeros((11, 11, 11))
        at = lambda d, o: tuple(5 + (o if 2 - i == d else 0) for i in range(3))  # noqa: E731
        for d in range(3):
            if d == ax:
                f[at(d, 1)] = -flip * x
                continue
            for o in range(-G, G + 1):
                w = UP[order].get(int(vs) * o, 0) if follow == "up" else KO[order][o + G]
                if w:
                    f[at(d, o)] = flip * (x if w > 0 else -x)
        sigma = 1.0
        D = np.full(3, float(x / float(KC[order]) * kap))     # kap near x, or far below u
        vet = np.full(3, vs * float(KC[order]) / kap)          # |vet| D near x
        out, fp = np.empty(1), np.empty(1)
        lib.fixed_advko(ax, order, _p(f), _p(vet), _p(D), ctypes.c_double(sigma), _p(out), _p(fp))
        tot = Fr(0)
        for d in range(3):
            u, k = Fr(float(abs(vet[d]) * D[d])), Fr(float(float(KC[order]) * sigma * D[d]))
            v = lambda o: Fr(float(f[at(d, o)]))  # noqa: E731
            if d == ax:
                tot += ({4: 16, 8: 768}[order] * u + {4: 32, 8: 512}[order] * k) * (v(1) - v(0))
                continue
            tot += u * sum(w * v(int(vs) * o) for o, w in UP[order].items())
            tot += k * sum(w * v(o - G) for o, w in enumerate(KO[order]))
        c = max(Fr(float(abs(vet[0]) * D[0])), Fr(float(float(KC[order]) * sigma * D[0])))
        bound = abs(tot) / 2 ** 53 + c * Fr(float(x)) * (weights * (Fr(1, 2 ** (52 + sh)) + Fr(1, 2 ** 58)) + last)
        assert abs(Fr(float(out[0])) - tot) <= bound, (x, follow, flip, vs, kap, out[0], float(tot))


@pytest.mark.parametrize("ax", [-1, 1, 2])
@pytest.mark.parametrize("order", [4, 8])
def test_negated_values_give_the_negated_sum(lib, order, ax):
    """Smooth fields: the bits of the sum with its sign flipped, so that a state with a reflection symmetry keeps it."""
    rng = np.random.default_rng(17 + order + ax)
    x = np.arange(11) - 5
    for _ in range(400):
        k, p = rng.uniform(0.02, 0.2, 3), rng.uniform(0, 6, 3)
        f = rng.uniform(-1, 1) + np.zeros((11, 11, 11))
        for d in range(3):
            f += np.cos(k[d] * x + p[d]).reshape([11 if 2 - i == d else 1 for i in range(3)])
        vet, D = rng.uniform(-0.1, 0.1, 3), 10.0 ** rng.uniform(-1, 1, 3)
        out = [np.empty(1), np.empty(1)]
        for o, s in zip(out, (1.0, -1.0)):
            lib.fixed_advko(ax, order, _p(np.ascontiguousarray(s * f)), _p(vet), _p(D), ctypes.c_double(0.3), _p(o), _p(np.empty(1)))
        assert out[0][0] == -out[1][0]


def test_subtraction_bound_and_ties(lib):
    """One rounding to nearest plus what the alignment cuts beyond 9 binades; ties away from zero, for either sign."""
    rng = np.random.default_rng(23)
    a = rng.uniform(0.5, 1, 4000) * rng.choice([-1.0, 1.0], 4000)
    b = rng.uniform(0.5, 1, 4000) * rng.choice([-1.0, 1.0], 4000) * 2.0 ** rng.integers(-70, 1, 4000)
    a[:4], b[:4] = (1.0, -1.0, 1.0, -1.0), (-2.0 ** -53, 2.0 ** -53, 2.0 ** -54, -2.0 ** -54)
    out = np.empty(4000)
    lib.fixed_sub(_p(a), _p(b), ctypes.c_long(4000), _p(out))
    for x, y, o in zip(a, b, out):
        exact, big = Fr(float(x)) - Fr(float(y)), max(abs(Fr(float(x))), abs(Fr(float(y))))
        assert abs(Fr(float(o)) - exact) <= abs(exact) / 2 ** 53 + big / 2 ** 61
    assert out[0] == 1.0 + 2.0 ** -52 and out[1] == -out[0] and out[2] == 1.0 and out[3] == -1.0


@pytest.mark.parametrize("ax", [-1, 1, 2])
@pytest.mark.parametrize("order", [4, 8])
def test_the_fp64_sum_that_takes_values_outside_the_range(lib, order, ax):
    """The merged FP64 stencil against rational arithmetic: at most 33 weights of up to four roundings each, summed in one
    chain, so 40 roundings of the terms' magnitudes bound it."""
    G = len(KO[order]) // 2
    rng = np.random.default_rng(29 + order + ax)
    for _ in range(60):
        f = np.ascontiguousarray(rng.uniform(-1, 1, (11, 11, 11)))
        vet, D, sigma = rng.uniform(-0.3, 0.3, 3), 10.0 ** rng.uniform(-1, 1, 3), 0.3
        out, fp = np.empty(1), np.empty(1)
        lib.fixed_advko(ax, order, _p(f), _p(vet), _p(D), ctypes.c_double(sigma), _p(out), _p(fp))
        tot, mag = Fr(0), Fr(0)
        for d in range(3):
            at = lambda o: Fr(float(f[tuple(5 + (o if 2 - i == d else 0) for i in range(3))]))  # noqa: E731
            u, k = Fr(float(abs(vet[d]) * D[d])), KC[order] * Fr(sigma) * Fr(float(D[d]))
            if d == ax:
                c = {4: 16, 8: 768}[order] * u + {4: 32, 8: 512}[order] * k
                tot += c * (at(1) - at(0))
                mag += c * (abs(at(1)) + abs(at(0)))
                continue
            s = 1 if vet[d] > 0 else -1
            terms = [u * w * at(s * o) for o, w in UP[order].items()] + [k * w * at(o - G) for o, w in enumerate(KO[order])]
            tot += sum(terms)
            mag += sum(abs(t) for t in terms)
        assert abs(Fr(float(fp[0])) - tot) <= 40 * mag / 2 ** 53
        assert abs(Fr(float(out[0])) - tot) <= 40 * mag / 2 ** 53
