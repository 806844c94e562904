"""FP32 rows with their own mesh on the warp-segment kernel, where its 32-bit positions,
its plain sums and its limiters could differ from the per-order kernels that hold 64-bit
positions and compensated sums: shifts of about one position unit, output cells over many
source cells, values that are not finite, and magnitudes far from 1."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _bump(n):
    return wl.bump_nodes(n, -np.pi, np.pi, 0.1387, 0.2773, 15.0)


def _plan(x, kernel=1, **kw):
    plan = ram.Plan([0, x.size - 1], x, **kw)
    assert plan.info().n_nseg_rows == 1
    t = plan.tuning()
    t.nonuniform_kernel_f32 = kernel
    plan.set_tuning(t)
    return plan


def _step(plan, q, s, dt=0.1, dv=None, scheme=ram.VANLEER, nsub=1, n_steps=1):
    a = torch.tensor(np.asarray(q), dtype=torch.float32, device=DEV)
    b = torch.empty_like(a)
    v0 = torch.tensor([s / dt], dtype=torch.float64, device=DEV)
    d = None if dv is None else torch.tensor(np.asarray(dv), dtype=torch.float32, device=DEV)
    ns = None if dv is None else torch.tensor([nsub], dtype=torch.int32, device=DEV)
    for _ in range(n_steps):
        ram.step(plan, a, b, v0, dt, dv=d, scheme=scheme, nsub=ns)
        a, b = b, a
    return a.double().cpu().numpy()


@pytest.mark.parametrize("units", [0.3, 0.8, 1.45, 2.55, 7.3])
@pytest.mark.parametrize("n", [510, 1533])
@pytest.mark.parametrize("order", [2, 3])
def test_shifts_of_about_one_position_unit(order, n, units):
    """A position unit is up to 2^-20 of the narrowest cell.  A top-hat of height 1 moved
    left by about that much puts s / dx into the empty cell beside its left end: one
    product and one quotient in FP32, within 1e-5 relative, and 1e-4 for what the oracle's
    FP64 positions leave of a shift of 1e-9 cells."""
    x = _bump(n)
    dx = np.diff(x)
    xc = 0.5 * (x[1:] + x[:-1])
    q = (np.abs(xc) < 0.08).astype(np.float64)  # its ends lie in the narrow cells
    beside = np.flatnonzero(q)[0] - 1
    s = -units * dx.min() * 2.0 ** -20
    got = _step(_plan(x, order=order), q, s)[beside]
    ref = oracle.step(x, q, oracle.shift_from_velocity(s / 0.1, 0.1), order, True)[beside]
    assert ref > 0.0
    assert abs(got - ref) <= 1e-4 * ref


@pytest.mark.parametrize("with_dv", [False, True])
def test_output_cells_over_many_source_cells(with_dv):
    """Wide cells over up to 144 narrow ones: their masses are sums of that many cells.
    Against the FP64 oracle on the same values, the wide cells within 2^-22 (products,
    their sum kept in two floats, one quotient: a few half units of 2^-24)."""
    rng = np.random.default_rng(8)
    w = np.ones(2000)
    w[1000:1010] = 140.0
    x = np.concatenate([[0.0], np.cumsum(w)]) / w.sum()
    n = w.size
    q = (1.0 + rng.random(n)).astype(np.float32).astype(np.float64)
    wide = np.flatnonzero(w > 1.0)
    dv = np.zeros(n) if with_dv else None
    for order in (2, 3):
        plan = _plan(x, order=order)
        for k in range(8):
            s = (1400.0 + 37.3 * k) / w.sum()  # under the wide cells: narrow ones
            got = _step(plan, q, s, dv=dv)
            ref = oracle.step(x, q, oracle.shift_from_velocity(s / 0.1, 0.1), order, True)
            err = np.abs(got - ref)[wide] / ref[wide]
            assert err.max() <= 2.0 ** -22, (order, k, err.max() * 2.0 ** 24)


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("order,limiter", [(2, True), (2, False), (3, True), (3, False),
                                           (4, True), (4, False)])
def test_values_that_are_not_finite(value, order, limiter):
    """A NaN reaches the cells that it reaches with the per-order kernel, an infinity none
    that neither of them reaches there; where both kernels' results are finite they
    agree."""
    n = 1533
    x = wl.random_nodes(n, seed=n + 5)
    q = 1.0 + np.random.default_rng(4).random(n)

    def run(kernel, v):
        plan = _plan(x, kernel, order=order, limiter=limiter)
        out = _step(plan, np.where(np.arange(n) == 700, v, q), 0.2)
        assert plan.check_errors() == 0
        return out

    got, ref, nan = run(1, value), run(0, value), run(0, np.nan)
    if np.isnan(value):
        np.testing.assert_array_equal(np.isfinite(got), np.isfinite(ref))
    assert not np.isfinite(got).all()
    assert np.isfinite(got[np.isfinite(nan) & np.isfinite(ref)]).all()
    fine = np.isfinite(got) & np.isfinite(ref)
    np.testing.assert_allclose(got[fine], ref[fine], rtol=1e-5)


@pytest.mark.parametrize("scale", [1e-30, 1e-24, 1.0, 1e30])
@pytest.mark.parametrize("length", [1e-9, 1.0, 1e13])
@pytest.mark.parametrize("order", [2, 3])
def test_magnitudes(order, length, scale):
    """Values and lengths far from 1: the step is linear in the values and does not depend
    on the unit of length (relative L1 against the FP64 oracle <= 1e-5)."""
    n = 777
    x = wl.random_nodes(n, seed=3) * length
    rng = np.random.default_rng(5)
    dx = np.diff(x)
    q = ((1.0 + rng.random(n)) * scale).astype(np.float32).astype(np.float64)
    dv = ((rng.random(n) - 0.5) * 1.6 * dx.min() / 0.1).astype(np.float32).astype(np.float64)
    s = 0.3217 * length
    plan = _plan(x, order=order)
    got = _step(plan, q, s, dv=dv)
    ref = oracle.step(x, q, oracle.shift_from_velocity(s / 0.1, 0.1), order, True, dv, 0.1,
                      ram.VANLEER, 1)
    assert plan.check_errors() == 0
    assert np.sum(np.abs(got - ref) / scale * dx) <= 1e-5 * np.sum(np.abs(ref) / scale * dx)


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("order", [2, 3])
def test_not_finite_with_a_residual(value, order):
    """Cells farther than the stencils of the shift and one van Leer sub-step (7 cells on
    each side) are as without the value, bit for bit."""
    n = 1533
    x = wl.random_nodes(n, seed=n + 5)
    rng = np.random.default_rng(4)
    q = 1.0 + rng.random(n)
    dv = (rng.random(n) - 0.5) * 0.6 * np.diff(x).min() / 0.1
    plan = _plan(x, order=order)
    s = 0.2 * (x[-1] - x[0])
    good = _step(plan, q, s, dv=dv)
    bad = _step(plan, np.where(np.arange(n) == 700, value, q), s, dv=dv)
    lo = np.searchsorted(x, x[700] + s) - 1
    hi = np.searchsorted(x, x[701] + s)
    assert not np.isfinite(bad[lo:hi]).all()
    far = np.ones(n, dtype=bool)
    far[lo - 7:hi + 7] = False
    np.testing.assert_array_equal(bad[far], good[far])
