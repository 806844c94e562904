"""The warp-segment transpose of uniform rows where its ranges end: rows of the
shortest length it takes, of one segment more or less, whole-cell and seam shifts,
one to eight sub-steps (the widest halo), arrays off the 16-byte boundary (the tiled
kernel), against the FP64 oracle at the suite's bars (relative L1 <= 1e-12 FP64,
1e-5 FP32)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_2305_05362_gb300 import ram, workloads as wl
from gpu_common import TOL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SHIFTS = [0.0, 3.0, 511.0, 0.4, 7.3, -1.25, 300.62]  # cells, one row each


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [508, 512, 516, 744, 748, 1000, 2052])
@pytest.mark.parametrize("order,nsub", [(2, 1), (3, 2), (4, 8), (3, 5), (3, 0)])
def test_matches_oracle(dtype, n, order, nsub):
    x = wl.uniform_nodes(n, 0.25, 2.0)
    rows = len(SHIFTS)
    plan = ram.Plan(np.arange(rows + 1) * n, x, order=order, limiter=False, shared_mesh=True)
    rng = np.random.default_rng(n + nsub)
    dt = 0.5
    dx = 2.0 / n

    def put(a, off=0):
        buf = torch.empty(a.size + off, dtype=dtype, device=DEV)[off:]
        return buf.copy_(torch.tensor(a, device=DEV))

    q, g = rng.standard_normal((2, rows * n))
    dv = (rng.random(rows * n) - 0.5) * 1.6 * max(nsub, 1) * dx / dt
    g0 = rng.standard_normal(rows * n)
    v0 = torch.tensor(np.array(SHIFTS) * dx / dt, device=DEV)
    ns = torch.full((rows,), max(nsub, 1), dtype=torch.int32, device=DEV)
    results = []
    for off in (0, 1):
        qd, gd, dvd, gdv = put(q, off), put(g), put(dv), put(g0)
        gin = torch.empty_like(gd)
        ram.step_adjoint(plan, qd, gd, gin, v0, dt, dv=dvd if nsub else None,
                         g_dv=gdv if nsub else None, nsub=ns)
        results.append((gin.double().cpu().numpy(), gdv.double().cpu().numpy()))
    tol = TOL["float64" if dtype == torch.float64 else "float32"]
    qr, gr, dvr, g0r = (t.double().cpu().numpy() for t in (put(q), put(g), put(dv), put(g0)))
    for r in range(rows):
        sl = slice(r * n, (r + 1) * n)
        ri, rd = oracle.step_adjoint(x, qr[sl], gr[sl], oracle.shift_from_velocity(float(v0[r]), dt),
                                     order, dvr[sl] if nsub else None, dt, max(nsub, 1))
        for gin, gdv in results:
            assert np.abs(gin[sl] - ri).sum() <= tol * np.abs(ri).sum(), r
            if nsub:
                ref = g0r[sl] + rd  # added into what was there
                assert np.abs(gdv[sl] - ref).sum() <= tol * (np.abs(g0r[sl]) + np.abs(rd)).sum(), r
    assert plan.check_errors() == 0


@pytest.mark.parametrize("n", [512, 515])
@pytest.mark.parametrize("k", [1, 2, 3, 6])
def test_steps_in_a_row_equal_single_calls(n, k):
    """ram.steps and ram.steps_adjoint give what k single calls give, bit for bit (also
    with an odd number of cells, where the kept states are padded)."""
    plan = ram.Plan([0, n, 2 * n], wl.uniform_nodes(n), order=3, limiter=False, shared_mesh=True)
    gen = torch.Generator(device=DEV).manual_seed(n + k)
    q, g, dv = torch.randn(3, 2 * n, generator=gen, device=DEV).unbind(0)
    dv = dv * (0.1 / n)
    v0 = torch.tensor([0.013, -0.4], dtype=torch.float64, device=DEV)
    out, g_in, g_dv = torch.empty_like(q), torch.empty_like(q), torch.ones_like(q)
    ram.steps(plan, q, out, k, v0, 1.0, dv=dv, scheme=ram.DONOR)
    ram.steps_adjoint(plan, q, g, g_in, k, v0, 1.0, dv=dv, g_dv=g_dv)
    states, gd = [q.contiguous()], torch.ones_like(q)
    for _ in range(k):
        nxt = torch.empty_like(states[-1])
        ram.step(plan, states[-1], nxt, v0, 1.0, dv=dv, scheme=ram.DONOR)
        states.append(nxt)
    assert torch.equal(out, states[-1])
    for i in reversed(range(k)):
        gi = torch.empty_like(q)
        ram.step_adjoint(plan, states[i], g, gi, v0, 1.0, dv=dv, g_dv=gd)
        g = gi
    # (a misaligned field takes the tiled kernel: the same numbers to rounding)
    close = dict(rtol=0, atol=0) if n % 4 == 0 else dict(rtol=1e-5, atol=1e-5)
    torch.testing.assert_close(g_in, g, **close)
    torch.testing.assert_close(g_dv, gd, **close)
    with pytest.raises(ram.RamError):
        ram.steps(plan, q, q, k, v0, 1.0, dv=dv)


@pytest.mark.parametrize("dt", [0.5, 1e-25, 1e-38, 1e35])
def test_shifts_beyond_two_float_range(dt):
    """FP32 rows whose shift, or a factor of it, two-float arithmetic does not hold to a
    fraction of a cell take the FP64 shift (the suite's FP32 bar; a fraction wrong by
    2^-10 of a cell, or a shift dropped, is far above it)."""
    n, order = 1024, 3
    x = wl.uniform_nodes(n, 0.0, 1.0)
    shifts = np.array([0.37, 2.0**20 - 0.4, 2.0**21 + 0.7, -3.3e7, 2.0**33 + 0.6, 2.0**41 + 0.3])
    rows = len(shifts)
    v0 = shifts / n / dt
    plan = ram.Plan(np.arange(rows + 1) * n, x, order=order, limiter=False, shared_mesh=True)
    rng = np.random.default_rng(5)
    q, g = (torch.tensor(a, dtype=torch.float32, device=DEV)
            for a in rng.standard_normal((2, rows * n)))
    gin = torch.empty_like(g)
    ram.step_adjoint(plan, q, g, gin, torch.tensor(v0, device=DEV), dt)
    assert plan.check_errors() == 0
    got, qr, gr = (t.double().cpu().numpy() for t in (gin, q, g))
    for r in range(rows):
        sl = slice(r * n, (r + 1) * n)
        ref, _ = oracle.step_adjoint(x, qr[sl], gr[sl], oracle.shift_from_velocity(v0[r], dt),
                                     order, None, dt, 1)
        assert np.abs(got[sl] - ref).sum() <= TOL["float32"] * np.abs(ref).sum(), r
