"""A residual velocity that is not a number spoils the cells around it (as in the oracle)
and nothing else: no Courant number is above 1, on any mesh, form or precision."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("mesh", ["uniform", "a4", "own"])
@pytest.mark.parametrize("scheme", [ram.DONOR, ram.VANLEER])
def test_no_cfl_error(dtype, mesh, scheme):
    n = 1024
    x = wl.random_nodes(n, seed=1) if mesh == "own" else wl.uniform_nodes(n)
    plan = ram.Plan([0, n], x, order=3, shared_mesh=True, a4=mesh == "a4")
    rng = np.random.default_rng(2)
    dv = (rng.random(n) - 0.5) * np.diff(x).min() / 0.1
    q = torch.tensor(1.0 + rng.random(n), dtype=dtype, device=DEV)
    v0 = torch.tensor([0.37], dtype=torch.float64, device=DEV)
    out = []
    for v in (dv[600], np.nan):
        d = torch.tensor(np.where(np.arange(n) == 600, v, dv), dtype=dtype, device=DEV)
        o = torch.empty_like(q)
        ram.step(plan, q, o, v0, 0.1, dv=d, scheme=scheme)
        assert plan.check_errors() == 0
        out.append(o.cpu().numpy())
    assert np.isnan(out[1][599:601]).all()
    far = np.abs(np.arange(n) - 599.5) > 3
    np.testing.assert_allclose(out[1][far], out[0][far], rtol=1e-13)
