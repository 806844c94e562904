"""The limited step does not depend on the unit of the values: the transpose linearised at
fields scaled by powers of two gives the same bits, on rows with their own mesh in FP32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("power", [-80, -60, 60])
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("with_dv", [False, True])
def test_power_of_two_values(power, order, with_dv):
    n = 1533
    x = wl.random_nodes(n, seed=7)
    plan = ram.Plan([0, n], x, order=order, adjoint=True)
    rng = np.random.default_rng(8)

    def put(a):
        return torch.tensor(a, dtype=torch.float32, device=DEV)

    q, g = put(1.0 + rng.random(n)), put(rng.random(n) - 0.5)
    dv = put((rng.random(n) - 0.5) * 1.6 * np.diff(x).min() / 0.1) if with_dv else None
    v0 = torch.tensor([3.217], dtype=torch.float64, device=DEV)
    out = []
    for scale in (1.0, 2.0 ** power):
        g_in = torch.empty_like(q)
        g_dv = torch.zeros_like(q) if with_dv else None
        ram.step_adjoint(plan, q * scale, g, g_in, v0, 0.1, dv=dv, g_dv=g_dv)
        out.append((g_in, g_dv / scale if with_dv else g_in))
    assert plan.check_errors() == 0
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])
