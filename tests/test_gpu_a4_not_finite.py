"""A value that is not finite in a step with the fourth-order correction reaches the cells
that it reaches with the separate kernels (arrays off the 16-byte boundary), 12 cells of
the inverse's weights and the stencils of the rest; cells beyond are as without it.  (The
separate kernels' FP32 residual there is the tiled one, whose sub-steps carry the value
less far than the ring kernel's: a stencil per sub-step is allowed for.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2305_05362_gb300 import ram, workloads as wl

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("limiter", [True, False])
@pytest.mark.parametrize("cells", [0.0, 7.3, -300.62])
@pytest.mark.parametrize("scheme,nsub", [(ram.VANLEER, 0), (ram.VANLEER, 1), (ram.DONOR, 3)])
def test_reach(dtype, value, limiter, cells, scheme, nsub):
    rows, n = 24, 1024
    plan = ram.Plan(np.arange(rows + 1) * n, wl.uniform_nodes(n), order=3, limiter=limiter,
                    shared_mesh=True, a4=True)
    rng = np.random.default_rng(nsub)
    good = 1.0 + rng.random(rows * n)
    dvn = (rng.random(rows * n) - 0.5) * 1.6 * max(nsub, 1) / n / 0.5
    bad = good.copy()
    # one in every row, over all positions in a lane and a segment
    at = np.array([(41 * r + 7) % n for r in range(rows)])
    bad[np.arange(rows) * n + at] = value
    v0 = torch.full((rows,), cells / n / 0.5, dtype=torch.float64, device=DEV)
    ns = torch.full((rows,), max(nsub, 1), dtype=torch.int32, device=DEV)

    def put(a, off=0):
        return torch.empty(a.size + off, dtype=dtype, device=DEV)[off:].copy_(
            torch.tensor(a, device=DEV))

    def run(q, off):
        qd, dv = put(q, off), put(dvn, off) if nsub else None
        out = torch.empty_like(put(q, off))
        ram.step(plan, qd, out, v0, 0.5, dv=dv, scheme=scheme, nsub=ns)
        return out.double().cpu().numpy().reshape(rows, n)

    got, ref, clean = run(bad, 0), run(bad, 1), run(good, 0)
    assert plan.check_errors() == 0
    lost, lost_ref = ~np.isfinite(got), ~np.isfinite(ref)
    dist = np.abs((np.arange(n)[None, :] - at[:, None] - round(cells) + n // 2) % n - n // 2)
    if dtype == torch.float64:
        np.testing.assert_array_equal(lost, lost_ref)
    else:
        allowed = lost_ref
        for _ in range(nsub * (2 if scheme == ram.VANLEER else 1)):
            allowed = allowed | np.roll(allowed, 1, 1) | np.roll(allowed, -1, 1)
        assert not (lost & ~allowed).any()
        # where a segment does not hold the value, the weights beyond 8 cells are left out
        assert (dist[lost_ref & ~lost] > 8).all()
    far = dist > 24
    # (fields of order 1; the forms that meet in a segment round differently)
    assert np.abs(got[far] - clean[far]).max() <= (1e-12 if dtype == torch.float64 else 1e-5)
