"""The radial sweep does not depend on the unit of length: radii and time step scaled by a
power of two give the same bits, at face areas far outside the range of FP32 too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("power", [-70, -20, 20, 70])
def test_power_of_two_units(dtype, power):
    nr, n = 21, 150
    plan = ram.Plan(np.arange(nr + 1) * n, wl.uniform_nodes(n), order=2, shared_mesh=True)
    rng = np.random.default_rng(2)
    q = torch.tensor(1.0 + rng.random(nr * n), dtype=dtype, device=DEV)
    vr = torch.tensor(rng.random((nr + 1) * n) - 0.5, dtype=dtype, device=DEV)
    rf = 0.4 + np.cumsum(0.05 + 0.05 * rng.random(nr + 1))
    out = []
    for scale in (1.0, 2.0 ** power):
        o = torch.empty_like(q)
        ram.radial_upwind(plan, q, o, torch.tensor(rf * scale, device=DEV), vr, 0.04 * scale,
                          scheme=ram.DONOR)
        out.append(o)
    assert plan.check_errors() == 0
    assert float((out[0] - q).abs().max()) > 1e-3
    assert torch.equal(out[0], out[1])
