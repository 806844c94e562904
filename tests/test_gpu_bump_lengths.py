"""Rings on the paper's bump mesh (16:1) at lengths where its narrow cells would fall below
2^20 position units of a full window: the FP32 warp-segment kernel takes them with a part
of its window, the FP64 one (64-bit positions) with all of it.  Against the FP64 oracle,
relative L1 <= 1e-12 (FP64) and 1e-5 (FP32) per row."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl
from gpu_common import TOL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
BUMP = (-np.pi, np.pi, 0.1387, 0.2773, 15.0)


def _check(dtype, x, q, out, shifts, order, dv, dt, scheme, nsub):
    dx, n = np.diff(x), x.size - 1
    for r, s in enumerate(shifts):
        sl = slice(r * n, (r + 1) * n)
        ref = oracle.step(x, q[sl], s, order, True, None if dv is None else dv[sl], dt, scheme,
                          max(nsub, 1))
        err = np.sum(np.abs(out[sl] - ref) * dx) / np.sum(np.abs(ref) * dx)
        assert err <= TOL[dtype], (r, err)


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("n", [511, 512, 640, 649, 650, 1024, 1290, 2048, 4096])
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("density", [True, False])
def test_one_step(dtype, n, order, density):
    t = getattr(torch, dtype)
    x = wl.bump_nodes(n, *BUMP)
    L, dx, dt = x[-1] - x[0], np.diff(x), 0.1
    cells = np.array([0.0, 0.4, 7.3, -31.9, 0.5 * n, 2.62 * n])
    rows = cells.size
    plan = ram.Plan(np.arange(rows + 1) * n, x, order=order, shared_mesh=True)
    if density:
        plan.set_density([BUMP])
    assert plan.info().n_nseg_rows == rows
    rng = np.random.default_rng(n + order)

    def put(a):
        return torch.tensor(a, dtype=t, device=DEV)

    q = put(1.0 + rng.random(rows * n))
    out = torch.empty_like(q)
    v0 = torch.tensor(cells * L / n / dt, dtype=torch.float64, device=DEV)
    shifts = [oracle.shift_from_velocity(v, dt) for v in v0.tolist()]
    for scheme, nsub in ((ram.VANLEER, 0), (ram.VANLEER, 1), (ram.VANLEER, 8), (ram.DONOR, 3)):
        dv = put((rng.random(rows * n) - 0.5) * 1.6 * nsub * dx.min() / dt) if nsub else None
        ns = torch.full((rows,), nsub, dtype=torch.int32, device=DEV) if nsub else None
        ram.step(plan, q, out, v0, dt, dv=dv, scheme=scheme, nsub=ns)
        _check(dtype, x, q.double().cpu().numpy(), out.double().cpu().numpy(), shifts, order,
               None if dv is None else dv.double().cpu().numpy(), dt, scheme, nsub)
    assert plan.check_errors() == 0


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("n", [512, 1533])
def test_thousand_steps(dtype, n):
    """A steady rotation of 1000 steps at the flat bars, and the mass: FP64 to 1e-13, FP32
    to 1e-6 (the rounding of the stored cells)."""
    x = wl.bump_nodes(n, *BUMP)
    dx, xc = np.diff(x), 0.5 * (x[1:] + x[:-1])
    plan = ram.Plan([0, n], x, order=3)
    assert plan.info().n_nseg_rows == 1
    q0 = (1.0 + 0.5 * np.sin(xc) + np.exp(-(xc / 0.2) ** 2)).astype(np.float32).astype(np.float64)
    a = torch.tensor(q0, dtype=getattr(torch, dtype), device=DEV)
    b = torch.empty_like(a)
    v0 = torch.tensor([3.31234 * 2.0 * np.pi / n / 0.1], dtype=torch.float64, device=DEV)
    ref = q0
    for _ in range(1000):
        ram.step(plan, a, b, v0, 0.1)
        a, b = b, a
        ref = oracle.step(x, ref, oracle.shift_from_velocity(v0.item(), 0.1), 3, True)
    out = a.double().cpu().numpy()
    assert plan.check_errors() == 0
    assert np.sum(np.abs(out - ref) * dx) <= TOL[dtype] * np.sum(np.abs(ref) * dx)
    assert abs(np.sum(out * dx) / np.sum(q0 * dx) - 1.0) <= (1e-13 if dtype == "float64" else 1e-6)
