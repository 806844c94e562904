"""FP32 rows on graded meshes and around the warp-segment kernel's window sizes: the
source window moves on where the mesh under a segment is finer than at it, halos
wider than the plan allows for cut a segment into pieces, and rows about as long as
one window take the period's other units.  Every step against the FP64 oracle at the
suite's FP32 bar (relative L1 <= 1e-5 per row)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl
from gpu_common import TOL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _nodes(mesh, n):
    if mesh == "bump":  # 16 : 1 over a short transition
        return wl.bump_nodes(n, -np.pi, np.pi, 0.1387, 0.2773, 15.0)
    if mesh == "geometric":  # widths from 1 to 8 and back
        t = np.abs(np.linspace(-1.0, 1.0, n))
        return np.concatenate([[0.0], np.cumsum(8.0 ** t)]) / np.sum(8.0 ** t)
    return wl.random_nodes(n, seed=n + 5)


@pytest.mark.parametrize("mesh", ["bump", "geometric", "random"])
@pytest.mark.parametrize("n", [152, 156, 160, 161, 162, 163, 164, 319, 330, 1533])
@pytest.mark.parametrize("order,limiter", [(2, True), (3, True), (4, False)])
def test_windows_and_halos(mesh, n, order, limiter):
    x = _nodes(mesh, n)
    L = x[-1] - x[0]
    rng = np.random.default_rng(n + order)
    q0 = (1.0 + rng.random(n)).astype(np.float32).astype(np.float64)
    plan = ram.Plan([0, n], x, order=order, limiter=limiter)
    assert plan.info().n_nseg_rows == 1 and plan.tuning().nonuniform_kernel_f32 == 1
    qd = torch.tensor(q0, dtype=torch.float32, device=DEV)
    out = torch.empty_like(qd)
    dx = np.diff(x)
    dt = 0.1
    for s in (0.0, 0.31 * L, -0.5 * L, 0.77 * L + 3.0 * L, 1e-3 * dx.min(), L - 1e-9 * L):
        for scheme, nsub in ((None, 0), (ram.VANLEER, 1), (ram.VANLEER, 8), (ram.DONOR, 3)):
            dv = None
            if nsub:
                dv = ((rng.random(n) - 0.5) * 1.6 * nsub * dx.min() / dt).astype(np.float32)
            v0 = torch.tensor([s / dt], dtype=torch.float64, device=DEV)
            ram.step(plan, qd, out, v0, dt,
                     dv=None if dv is None else torch.tensor(dv, device=DEV),
                     scheme=ram.VANLEER if scheme is None else scheme,
                     nsub=torch.tensor([nsub], dtype=torch.int32, device=DEV) if nsub else None)
            torch.cuda.synchronize()
            ref = oracle.step(x, q0, oracle.shift_from_velocity(s / dt, dt), order, limiter,
                              None if dv is None else dv.astype(np.float64), dt,
                              ram.VANLEER if scheme is None else scheme, max(nsub, 1))
            err = np.sum(np.abs(out.double().cpu().numpy() - ref) * dx) / np.sum(np.abs(ref) * dx)
            assert err <= TOL["float32"], (s, scheme, nsub, err)
    assert plan.check_errors() == 0
