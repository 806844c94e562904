"""The transpose of uniform rows where the cotangent, the input or the residual velocity
holds a value that is not finite, or the velocity zeros of either sign: the warp-segment
kernel's gradients are not finite where the tile passes' are not (arrays off the 16-byte
boundary), and agree elsewhere."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("where", ["g_out", "q_in", "dv"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("order,nsub", [(2, 1), (3, 1), (3, 3), (4, 2)])
def test_same_cells_as_the_tile_passes(dtype, where, value, order, nsub):
    rows, n = 24, 1024
    plan = ram.Plan(np.arange(rows + 1) * n, wl.uniform_nodes(n), order=order, limiter=False,
                    shared_mesh=True)
    rng = np.random.default_rng(order + nsub)
    a = {"g_out": rng.random(rows * n) - 0.5, "q_in": 1.0 + rng.random(rows * n),
         "dv": (rng.random(rows * n) - 0.5) * 1.6 * nsub / n / 0.5}
    at = np.array([(41 * r + 7) % n for r in range(rows)])
    a["dv"][::11] = 0.0
    a["dv"][::13] = -0.0
    a[where][np.arange(rows) * n + at] = value
    v0 = torch.tensor((rng.random(rows) - 0.5) * 40.0 / n / 0.5, device=DEV)
    ns = torch.full((rows,), nsub, dtype=torch.int32, device=DEV)

    def put(x, off):
        return torch.empty(x.size + off, dtype=dtype, device=DEV)[off:].copy_(
            torch.tensor(x, device=DEV))

    out = []
    for off in (0, 1):
        t = {k: put(v, off) for k, v in a.items()}
        g_in, g_dv = put(np.zeros(rows * n), off), put(np.zeros(rows * n), off)
        ram.step_adjoint(plan, t["q_in"], t["g_out"], g_in, v0, 0.5, dv=t["dv"], g_dv=g_dv, nsub=ns)
        out.append([g.double().cpu().numpy() for g in (g_in, g_dv)])
    tol = 1e-12 if dtype == torch.float64 else 1e-5
    for got, ref in zip(*out):
        fine = np.isfinite(ref)
        np.testing.assert_array_equal(np.isfinite(got), fine)
        scale = np.abs(ref[fine]).max()
        assert np.abs(got[fine] - ref[fine]).max() <= tol * scale
