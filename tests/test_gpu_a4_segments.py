"""The fourth-order cell-average correction inside the warp-segment kernels where their
ranges end: rows of one segment more or less, whole-cell and seam shifts, up to eight
sub-steps, and arrays off the 16-byte boundary (the separate kernels), against the
FP64 oracle (relative L1 <= 1e-12 FP64, 1e-5 FP32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl
from gpu_common import TOL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SHIFTS = np.array([0.0, 3.0, -511.0, 0.4, 7.3, 300.62])  # cells, one row each


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [508, 512, 516, 700, 720, 2052])
@pytest.mark.parametrize("limiter", [True, False])
@pytest.mark.parametrize("scheme,nsub", [(1, 0), (1, 1), (0, 3), (1, 8)])
def test_matches_oracle(dtype, n, limiter, scheme, nsub):
    rows = SHIFTS.size
    x = wl.uniform_nodes(n, 0.25, 2.0)
    plan = ram.Plan(np.arange(rows + 1) * n, x, order=3, limiter=limiter, shared_mesh=True, a4=True)
    rng = np.random.default_rng(n + nsub)
    dx, dt = 2.0 / n, 0.5
    q = 1.0 + rng.random(rows * n)
    dv = (rng.random(rows * n) - 0.5) * 1.6 * max(nsub, 1) * dx / dt
    v0 = torch.tensor(SHIFTS * dx / dt, device=DEV)
    ns = torch.full((rows,), max(nsub, 1), dtype=torch.int32, device=DEV)

    def put(a, off=0):
        return torch.empty(a.size + off, dtype=dtype, device=DEV)[off:].copy_(
            torch.tensor(a, device=DEV))

    dvd = put(dv)
    outs = []
    for off in (0, 1):
        qd = put(q, off)
        out = torch.empty_like(qd)
        ram.step(plan, qd, out, v0, dt, dv=dvd if nsub else None, scheme=scheme, nsub=ns)
        outs.append(out.double().cpu().numpy())
    assert plan.check_errors() == 0
    qr, dvr = put(q).double().cpu().numpy(), dvd.double().cpu().numpy()
    tol = TOL["float64" if dtype == torch.float64 else "float32"]
    for r in range(rows):
        sl = slice(r * n, (r + 1) * n)
        ref = oracle.step_a4(x, qr[sl], oracle.shift_from_velocity(float(v0[r]), dt), limiter,
                             dvr[sl] if nsub else None, dt, scheme, max(nsub, 1))
        for out in outs:
            assert np.abs(out[sl] - ref).sum() <= tol * np.abs(ref).sum(), r


@pytest.mark.parametrize("case", ["huge", "nan"])
def test_fp64_values_out_of_the_ordinary(case):
    """Against the separate kernels (arrays off the 16-byte boundary), whose limiters
    compare in floating point."""
    n = 1024
    plan = ram.Plan([0, n], wl.uniform_nodes(n), order=3, shared_mesh=True, a4=True)
    q = 1.0 + np.random.default_rng(1).random(n)
    if case == "huge":
        q *= 2.0 ** 1003
    else:
        q[300] = np.nan
    v0 = torch.tensor([7.3 / n], dtype=torch.float64, device=DEV)
    outs = []
    for off in (0, 1):
        qd = torch.empty(n + off, dtype=torch.float64, device=DEV)[off:].copy_(
            torch.tensor(q, device=DEV))
        out = torch.empty_like(qd)
        ram.step(plan, qd, out, v0, 1.0)
        outs.append(out)
    fine = torch.isfinite(outs[0]) & torch.isfinite(outs[1])
    assert int(fine.sum()) >= (n if case == "huge" else n - 2 * 60)
    torch.testing.assert_close(outs[0][fine], outs[1][fine], rtol=1e-12, atol=0.0)
    if case == "nan":
        # (the recursions carry it to their segment's end, the separate kernel 12 cells)
        assert not bool(torch.isfinite(outs[0][307:309]).any())
