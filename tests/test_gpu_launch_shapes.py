"""The launch shapes of the right-hand side (tiles spread over four warps, three or four blocks per SM; one point per
thread, two or four blocks per SM) on sizes at the lines of the rule that chooses among them: two steps, bitwise
against the same grid in a batch with a tile shape set, which always runs one point per thread, and one evaluation of
the right-hand side against the oracle.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.oracle import Oracle  # noqa: E402
from paper_2505_00097_gb300 import binding as B  # noqa: E402
from paper_2505_00097_gb300 import build as BUILD  # noqa: E402
from paper_2505_00097_gb300 import workloads as W  # noqa: E402
from tests._common import assert_close  # noqa: E402

pytestmark = pytest.mark.gpu

KO8 = [0.3] * 17 + [0.99] * 7
KINDS = {
    "cyl_two_point": lambda n: W.sinh_cylindrical((33, 2, max(12, n // 66)), rho_max=30.0, z_max=30.0),
    "sph_two_point": lambda n: W.sinh_spherical((33, max(10, n // 66), 2)),
    "sph_general": lambda n: W.sinh_spherical((33, max(6, n // 792), 24)),
    "cyl_general": lambda n: W.sinh_cylindrical((33, 6, max(12, n // 198)), rho_max=30.0, z_max=30.0),
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    BUILD.build()
    B.lib()


# tiles of 32 points per SM: below and above one round of three and of four spread blocks, two rounds of three, one round
# of two blocks of 128 points, three of them with the outer blocks on top, and more
@pytest.mark.parametrize("per_sm", [0.2, 2.8, 3.1, 3.95, 4.3, 6.2, 8.3, 11.95, 13.0])
@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("order", [4, 8])
def test_every_shape_computes_the_same_bits(order, kind, per_sm):
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    spec = KINDS[kind](int(32 * per_sm * sm))
    if order == 8:
        spec = dict(spec, NG=5, ko_sigma=KO8)
    out = []
    for batched in (False, True):
        g = B.Grid(spec)
        g.set_brill_lindquist((0.6, 0.4), ((0, 0, 0.4), (0, 0, -0.6)), 1e-6, 3)
        if batched:
            b = B.Batch([g])
            b.set_tile(32, 4)
            (b.ssprk3_step if order == 8 else b.rk4_step)([g.dt_cfl], 2)
        else:
            (g.ssprk3_step if order == 8 else g.rk4_step)(g.dt_cfl, 2)
        y = np.empty(24 * g.T)
        g.get_state(y, True)
        out.append(y)
        if batched:
            b.close()
        g.close()
    assert np.all(np.isfinite(out[0])) and np.array_equal(out[0], out[1])


# grids of uneven sizes, tiles per SM of the whole batch: one round of three and of four spread blocks, two rounds of
# three, one point per thread with two and with four blocks per SM
@pytest.mark.parametrize("choice", ["default", "autotune"])
@pytest.mark.parametrize("per_sm", [0.5, 3.6, 5.2, 7.0, 13.0])
@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("order", [4, 8])
def test_a_batch_of_any_shape_computes_the_bits_of_its_grids(order, kind, per_sm, choice):
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    specs = [KINDS[kind](int(32 * per_sm * sm * w)) for w in (0.2, 0.5, 0.3)]
    if order == 8:
        specs = [dict(s, NG=5, ko_sigma=KO8) for s in specs]
    out = []
    for batched in (False, True):
        grids = [B.Grid(s) for s in specs]
        for q, g in enumerate(grids):
            g.set_brill_lindquist((0.6, 0.4), ((0, 0, 0.4), (0, 0, -0.6)), 1e-6, 3 + q)
        dts = [g.dt_cfl for g in grids]
        if batched:
            b = B.Batch(grids)
            if choice == "autotune":
                b.autotune(dts)
            (b.ssprk3_step if order == 8 else b.rk4_step)(dts, 2)
        else:
            for g, dt in zip(grids, dts):
                (g.ssprk3_step if order == 8 else g.rk4_step)(dt, 2)
        for g in grids:
            y = np.empty(24 * g.T)
            g.get_state(y, True)
            out.append(y)
        if batched:
            b.close()
        for g in grids:
            g.close()
    for a, c in zip(out[:3], out[3:]):
        assert np.all(np.isfinite(a)) and np.array_equal(a, c)


@pytest.mark.parametrize("per_sm", [2.8, 3.1, 4.3, 8.3, 13.0])
@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("order", [4, 8])
def test_one_evaluation_of_every_shape_matches_the_oracle(order, kind, per_sm):
    """1e-12 of the largest component of each tensor, as every right-hand-side parity test."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    spec = KINDS[kind](int(32 * per_sm * sm))
    if order == 8:
        spec = dict(spec, NG=5, ko_sigma=KO8)
    o = Oracle(spec)
    y = W.random_state(o.n, seed=31, smooth=True)
    o.inner_bc(y)
    g = B.Grid(spec)
    out = torch.zeros(y.size, dtype=torch.float64, device="cuda")
    g.rhs(torch.from_numpy(y).cuda(), out)
    torch.cuda.synchronize()
    assert_close(out.cpu().numpy(), o.rhs(y), o.T, 1e-12, mask=o.interior_mask(), what=f"{kind} {order}")
    g.close()


# one round of three, four and six spread blocks per SM, one of three blocks of 128 points, and more
@pytest.mark.parametrize("per_sm", [0.2, 2.9, 3.6, 5.5, 8.0, 13.0])
@pytest.mark.parametrize("kind", ["cyl_two_point", "sph_general"])
@pytest.mark.parametrize("order", [4, 8])
def test_the_constraints_of_every_shape_match_the_oracle(order, kind, per_sm):
    """Values to 1e-12 of the largest, norms to 1e-10, as every parity test of the constraints."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    spec = KINDS[kind](int(32 * per_sm * sm))
    if order == 8:
        spec = dict(spec, NG=5, ko_sigma=KO8)
    o = Oracle(spec)
    y = W.random_state(o.n, seed=41, smooth=True)
    o.inner_bc(y)
    m = o.interior_mask()
    g = B.Grid(spec)
    yd = torch.from_numpy(y).cuda()
    for comps, fn, ref in ((1, g.hamiltonian, o.hamiltonian(y)), (3, g.momentum, o.momentum(y))):
        out = torch.zeros(comps * o.T, dtype=torch.float64, device="cuda")
        norms = fn(yd, out)
        torch.cuda.synchronize()
        got, want = out.cpu().numpy().reshape(comps, o.T)[:, m], np.asarray(ref[0]).reshape(comps, o.T)[:, m]
        assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
        for a, b in zip(norms, ref[-3:-1]):   # l2, linf
            assert abs(a - b) <= 1e-10 * abs(b)
    g.close()
