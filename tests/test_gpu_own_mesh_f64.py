"""FP64 rows with their own mesh on the warp-segment kernel: graded meshes whose source
windows move on, rows around the window's length (the halved position units), halos
that cut a segment into pieces, and values its bit-level comparisons do not cover,
against the FP64 oracle (relative L1 <= 1e-12 per row)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _nodes(mesh, n):
    if mesh == "bump":
        return wl.bump_nodes(n, -np.pi, np.pi, 0.1387, 0.2773, 15.0)
    if mesh == "geometric":
        t = np.abs(np.linspace(-1.0, 1.0, n))
        return np.concatenate([[0.0], np.cumsum(8.0 ** t)]) / np.sum(8.0 ** t)
    return wl.random_nodes(n, seed=n + 5)


def _step(plan, q, s, dt, dv, scheme, nsub):
    qd = torch.tensor(q, device=DEV)
    out = torch.empty_like(qd)
    ram.step(plan, qd, out, torch.tensor([s / dt], dtype=torch.float64, device=DEV), dt,
             dv=None if dv is None else torch.tensor(dv, device=DEV), scheme=scheme,
             nsub=None if dv is None else torch.tensor([nsub], dtype=torch.int32, device=DEV))
    return out.cpu().numpy()


@pytest.mark.parametrize("mesh", ["bump", "geometric", "random"])
@pytest.mark.parametrize("n", [34, 152, 160, 163, 164, 319, 330, 1533])
@pytest.mark.parametrize("order,limiter", [(2, True), (2, False), (3, True), (3, False),
                                           (4, True), (4, False)])
def test_windows_and_halos(mesh, n, order, limiter):
    x = _nodes(mesh, n)
    L, dx, dt = x[-1] - x[0], np.diff(x), 0.1
    rng = np.random.default_rng(n + order)
    q = 1.0 + rng.random(n)
    q[:9] = 1.5  # a flat stretch
    plan = ram.Plan([0, n], x, order=order, limiter=limiter)
    for s in (0.0, 0.31 * L, -0.5 * L, 3.77 * L, 1e-3 * dx.min(), L - 1e-9 * L):
        for scheme, nsub in ((ram.VANLEER, 0), (ram.VANLEER, 1), (ram.VANLEER, 8), (ram.DONOR, 3)):
            dv = (rng.random(n) - 0.5) * 1.6 * nsub * dx.min() / dt if nsub else None
            out = _step(plan, q, s, dt, dv, scheme, nsub)
            ref = oracle.step(x, q, oracle.shift_from_velocity(s / dt, dt), order, limiter, dv, dt,
                              scheme, max(nsub, 1))
            err = np.sum(np.abs(out - ref) * dx) / np.sum(np.abs(ref) * dx)
            assert err <= 1e-12, (s, scheme, nsub, err)
    assert plan.check_errors() == 0


@pytest.mark.parametrize("scale", [1e-130, 0.0])
@pytest.mark.parametrize("order", [2, 3])
def test_magnitudes(scale, order):
    n = 1533
    x = _nodes("random", n)
    q = (1.0 + np.random.default_rng(3).random(n)) * scale
    plan = ram.Plan([0, n], x, order=order)
    out = _step(plan, q, 0.123, 0.1, None, ram.VANLEER, 1)
    ref = oracle.shift(x, q, oracle.shift_from_velocity(0.123 / 0.1, 0.1), order, True)
    assert np.sum(np.abs(out / max(scale, 1e-300) - ref / max(scale, 1e-300))) <= 1e-12 * n


@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("order,with_dv", [(2, False), (3, True)])
def test_a_value_that_is_not_finite_stays_where_it_is(value, order, with_dv):
    """The cells the value reaches are not finite; those farther than the stencils of the
    shift and one van Leer sub-step (7 cells on each side) are as without it."""
    n = 1533
    x = _nodes("random", n)
    rng = np.random.default_rng(4)
    q = 1.0 + rng.random(n)
    dv = (rng.random(n) - 0.5) * 0.6 * np.diff(x).min() / 0.1 if with_dv else None
    plan = ram.Plan([0, n], x, order=order)
    s = 0.2 * (x[-1] - x[0])
    good = _step(plan, q, s, 0.1, dv, ram.VANLEER, 1)
    bad_q = q.copy()
    bad_q[700] = value
    bad = _step(plan, bad_q, s, 0.1, dv, ram.VANLEER, 1)
    lo = np.searchsorted(x, x[700] + s) - 1
    hi = np.searchsorted(x, x[701] + s)
    assert not np.isfinite(bad[lo:hi]).all()
    far = np.ones(n, dtype=bool)
    far[lo - 7:hi + 7] = False
    # (a window that holds the value decides its limiters in floating point)
    np.testing.assert_allclose(bad[far], good[far], rtol=1e-13)
