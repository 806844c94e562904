"""The transpose on rows of a few cells, where a shifted cell may begin and end in the same
output cell with all the others in between; against the FP64 oracle (relative L1 <= 1e-11:
the values that cancel are a few, so the suite's 1e-12 with a digit to spare)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 9])
@pytest.mark.parametrize("order,limiter", [(2, True), (2, False), (3, True), (3, False), (4, False)])
def test_own_mesh(n, order, limiter):
    rng = np.random.default_rng(10 * n + order)

    def put(a):
        return torch.tensor(a, dtype=torch.float64, device=DEV)

    for k in range(40):
        x = wl.random_nodes(n, 97 * n + k, ratio=6.0)
        plan = ram.Plan([0, n], x, order=order, limiter=limiter, adjoint=True)
        q, g, s = 1.0 + rng.random(n), rng.random(n) - 0.5, float(rng.uniform(-2.0, 2.0))
        g_in = put(np.zeros(n))
        ram.step_adjoint(plan, put(q), put(g), g_in, put([s / 0.1]), 0.1)
        sh = oracle.shift_from_velocity(s / 0.1, 0.1)
        ref = (oracle.step_adjoint_limited(x, q, g, sh, order, True) if limiter
               else oracle.step_adjoint(x, q, g, sh, order))[0]
        assert np.abs(g_in.cpu().numpy() - ref).sum() <= 1e-11 * np.abs(ref).sum(), (k, s)
        assert plan.check_errors() == 0


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("limiter", [True, False])
@pytest.mark.parametrize("nsub", [1, 8])
def test_velocity_gradient_cancels(dtype, limiter, nsub):
    """At rest over a field of ones the gradient of interface j is dt times the difference of
    the cotangent over the widths, each cell's rounded alike on its two sides: one cell
    gives 0, two give opposite values, bit for bit."""
    rng = np.random.default_rng(5)

    def put(a, t=dtype):
        return torch.tensor(a, dtype=t, device=DEV)

    for k in range(40):
        for n in (1, 2):
            x = wl.random_nodes(n, 31 * n + k, ratio=3.0)
            plan = ram.Plan([0, n], x, order=3, limiter=limiter, adjoint=True)
            g_in, g_dv = put(np.zeros(n)), put(np.zeros(n))
            ram.step_adjoint(plan, put(np.ones(n)), put(rng.random(n) - 0.5), g_in,
                             put([0.0], torch.float64), 0.1, dv=put(np.zeros(n)), g_dv=g_dv,
                             nsub=put([nsub], torch.int32))
            assert float(g_dv.sum()) == 0.0
            assert n == 1 or float(g_dv.abs().max()) > 0.0
