"""The tiled own-mesh kernels (k_general with a residual, k_gwarp without) on the rows that
reach them: one cell 200 times as wide as the others, more source cells than a window of
the warp-segment kernels holds (tests/test_segments.py), in both precisions; and the FP32
scan, by tuning.  Against the FP64 oracle (relative L1 <= 1e-12 FP64, 1e-5 FP32)."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl
from gpu_common import TOL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
DT = {"float64": torch.float64, "float32": torch.float32}


def _crowded(n, seed):
    """Nodes of a row whose cell n // 3 lies over about 200 of the others."""
    w = np.exp(np.random.default_rng(seed).uniform(math.log(0.8), math.log(1.25), n))
    w[n // 3] = 200.0
    return np.concatenate([[0.0], np.cumsum(w)]) / w.sum()


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("n,order,limiter",  # one tile, one or two, windowed tiles
                         [(n, o, lim) for n in (220, 700, 20000)
                          for o, lim in ((2, True), (2, False), (3, True), (3, False), (4, True))]
                         + [(20000, 4, False)])
def test_crowded_rows(dtype, n, order, limiter):
    """Smooth fields (white noise would show the oracle's own rounding of x - s, 1e-11 of a
    cell at 20000 cells); flat beside the wide cell for order 4, whose weights there amplify
    any rounding by 1e3 (unlimited on the long row alone, where few cells are near it)."""
    x = _crowded(n, n + order)
    dx, dt = np.diff(x), 0.1
    plan = ram.Plan([0, n], x, order=order, limiter=limiter)
    plan.set_tiling(512, 128)
    assert plan.info().n_nseg_rows == 0
    assert n < 1000 or plan.info().n_tiles_general > 20
    rng = np.random.default_rng(n)
    q = wl.three_gaussians(x, n)
    if order == 4:
        q[n // 3 - 8:n // 3 + 9] = 1.5
    qd = torch.tensor(q, dtype=DT[dtype], device=DEV)
    q = qd.double().cpu().numpy()
    out = torch.empty_like(qd)
    for s in (0.0, 0.3 * dx.min(), 123.4 / n, 0.5, -2.0 - 17.3 / n):
        for scheme, nsub in ((ram.VANLEER, 0), (ram.VANLEER, 1), (ram.VANLEER, 8), (ram.DONOR, 3)):
            dv = None
            if nsub:
                dv = torch.tensor((rng.random(n) - 0.5) * 1.6 * nsub * dx.min() / dt,
                                  dtype=DT[dtype], device=DEV)
            v0 = torch.tensor([s / dt], dtype=torch.float64, device=DEV)
            ram.step(plan, qd, out, v0, dt, dv=dv, scheme=scheme,
                     nsub=torch.tensor([nsub], dtype=torch.int32, device=DEV) if nsub else None)
            ref = oracle.step(x, q, oracle.shift_from_velocity(s / dt, dt), order, limiter,
                              None if dv is None else dv.double().cpu().numpy(), dt, scheme,
                              max(nsub, 1))
            err = np.sum(np.abs(out.double().cpu().numpy() - ref) * dx) / np.sum(np.abs(ref) * dx)
            assert err <= TOL[dtype], (s, scheme, nsub, err)
    assert plan.check_errors() == 0


def test_step_scan_is_compensated_on_the_tiled_kernel():
    """The prefix sum of the tiled kernel (FP32 cells): one row of 65536 cells, PPM with a
    residual, a shift of 300 cells, tiles of 2048.  Every output mass is a difference of
    two window prefix sums over up to 2400 cells: a plain FP32 running sum would err by
    up to 1e-4 of a cell's mass, the two-float scan leaves the rounding of the
    reconstruction and the output.  Relative L1 <= 1e-6."""
    n = 65536
    x = wl.random_nodes(n, seed=41, ratio=4.0)
    xc = 0.5 * (x[1:] + x[:-1])
    q = 1.0 + 0.5 * np.sin(2 * math.pi * 3 * xc) + np.exp(-((xc - 0.4) / 0.05) ** 2)
    qd = torch.tensor(q, dtype=torch.float32, device=DEV)
    dvd = torch.tensor(0.002 * np.sin(2 * math.pi * 5 * x[:-1]), dtype=torch.float32, device=DEV)
    plan = ram.Plan([0, n], x, order=3, limiter=True)
    t = plan.tuning()
    t.nonuniform_kernel_f32, t.tile_cells, t.threads = 0, 2048, 512
    plan.set_tuning(t)
    dt = 1e-3
    v0 = torch.tensor([300.0 / n / dt], dtype=torch.float64, device=DEV)
    out = torch.empty_like(qd)
    ram.step(plan, qd, out, v0, dt, dv=dvd, scheme=ram.VANLEER)
    assert plan.check_errors() == 0
    ref = oracle.step(x, qd.double().cpu().numpy(), oracle.shift_from_velocity(v0.item(), dt), 3,
                      True, dvd.double().cpu().numpy(), dt, oracle.VANLEER, 1)
    got = out.double().cpu().numpy()
    assert np.abs(got - ref).sum() <= 1e-6 * np.abs(ref).sum()
