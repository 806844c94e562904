"""The FP64 warp-segment kernel where its forms end: rows of one segment more or less,
whole-cell and seam shifts, up to eight sub-steps, every order and limiter, against
the FP64 oracle (relative L1 <= 1e-12); and values that its bit-level comparisons do
not cover (very large and very small ones, infinities, NaN), against the persistent
whole-row kernel, which compares in floating point."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SHIFTS = np.array([0.0, 3.0, -511.0, 0.4, 7.3, -1.25, 300.62])  # cells, one row each


def _plan(n, order, limiter, kernel=1):
    rows = SHIFTS.size
    plan = ram.Plan(np.arange(rows + 1) * n, wl.uniform_nodes(n, 0.25, 2.0), order=order,
                    limiter=limiter, shared_mesh=True)
    t = plan.tuning()
    t.uniform_kernel_f64 = kernel
    plan.set_tuning(t)
    return plan


def _step(plan, q, dv, dx, scheme, nsub):
    dt = 0.5
    out = torch.empty_like(q)
    ns = torch.full((plan.n_rows,), max(nsub, 1), dtype=torch.int32, device=DEV)
    ram.step(plan, q, out, torch.tensor(SHIFTS * dx / dt, device=DEV), dt,
             dv=dv if nsub else None, scheme=scheme, nsub=ns)
    return out


@pytest.mark.parametrize("n", [512, 514, 740, 752, 2050])
@pytest.mark.parametrize("order,limiter", [(2, True), (2, False), (3, True), (3, False),
                                           (4, False)])
@pytest.mark.parametrize("scheme,nsub", [(1, 0), (1, 1), (1, 3), (0, 5), (1, 8)])
def test_matches_oracle(n, order, limiter, scheme, nsub):
    rng = np.random.default_rng(n + order + nsub)
    dx, dt = 2.0 / n, 0.5
    q = 1.0 + rng.random(SHIFTS.size * n)
    q[n // 2:n // 2 + 40] = 1.0  # a flat stretch: zero differences
    dv = (rng.random(q.size) - 0.5) * 1.6 * max(nsub, 1) * dx / dt
    plan = _plan(n, order, limiter)
    out = _step(plan, torch.tensor(q, device=DEV), torch.tensor(dv, device=DEV), dx, scheme,
                nsub).cpu().numpy()
    assert plan.check_errors() == 0
    x = wl.uniform_nodes(n, 0.25, 2.0)
    for r, s in enumerate(SHIFTS):
        sl = slice(r * n, (r + 1) * n)
        ref = oracle.step(x, q[sl], oracle.shift_from_velocity(s * dx / dt, dt), order, limiter,
                          dv[sl] if nsub else None, dt, scheme, max(nsub, 1))
        assert np.abs(out[sl] - ref).sum() <= 1e-12 * np.abs(ref).sum(), r


@pytest.mark.parametrize("case", ["huge", "tiny", "inf", "nan", "nan_dv", "cfl"])
@pytest.mark.parametrize("order", [2, 3, 4])
def test_values_out_of_the_ordinary(case, order):
    n, nsub = 1024, 2
    dx = 2.0 / n
    rng = np.random.default_rng(order)
    q = 1.0 + rng.random(SHIFTS.size * n)
    dv = (rng.random(q.size) - 0.5) * 0.8 * nsub * dx / 0.5
    if case == "huge":
        q[n:2 * n] *= 1e302
    elif case == "tiny":
        q *= 1e-290
    elif case == "cfl":
        dv[5 * n + 17] *= 40.0
    elif case == "nan_dv":
        dv[3 * n + 100] = np.nan
    else:
        q[[100, 2 * n + 511, 4 * n]] = np.inf if case == "inf" else np.nan
    qd, dvd = torch.tensor(q, device=DEV), torch.tensor(dv, device=DEV)
    outs, status = [], []
    for kernel in (1, 0):
        plan = _plan(n, order, order != 4, kernel)
        outs.append(_step(plan, qd, dvd, dx, ram.VANLEER, nsub))
        status.append(plan.check_errors())
    assert status[0] == status[1] == (3 if case == "cfl" else 0)
    torch.testing.assert_close(outs[0], outs[1], rtol=1e-12, atol=0.0, equal_nan=True)
