"""The work whose speed counts: what programs have this package do, over its real range.

Every case is one pass through the public entry points (ram.step, ram.shift, ram.step_2d,
autograd.rollout) on a plan as the program keeps it, with the plan's default launch
shapes.  The families, told apart by "kind":

  disk     a polar disk's azimuthal sweep: every ring a periodic row of equal cells on one
           shared mesh, Keplerian shift, 1% residual velocity sub-cycled per ring.
  rows     a batch of independent rows of uneven lengths, each on its own non-uniform mesh
           (n_rows = 1: a line), with or without a residual velocity.
  disk2d   the dimensionally split step of a polar disk on the bump mesh of the paper's
           two-dimensional runs: the azimuthal step, then the radial sweep.
  adjoint  a differentiable rollout: the loss of the final field against a target, its
           gradients with respect to the initial field and the residual velocity.
  a4       the disk's step with the fourth-order cell-average correction (point values).

exact() restates the method in plain FP64 torch: the shift as differences of the
cumulative mass at the shifted nodes, the residual sub-steps with rolled arrays, the
gradients by torch's own differentiation.
"""
import math

import numpy as np
import torch

from paper_2305_05362_gb300 import autograd, ram, workloads

DEV = "cuda:0"
DTYPES = {"f32": torch.float32, "f64": torch.float64}
MAX_CELLS = 8192 * 16384


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # a single line, the smallest problem that is stepped in earnest: latency
        {"name": "line_4096", "kind": "rows", "n_rows": 1, "n_min": 4096, "n_max": 4096,
         "orders": "3", "limiter": True, "dv": True, "entry": "step", "dtype": "f32"},
        # a small disk, as parameter studies run by the thousand: launches and latency
        {"name": "disk_64x512", "kind": "disk", "n_r": 64, "n_phi": 512, "order": 3,
         "limiter": True, "dtype": "f32"},
        # the default disk of the benchmark: the ordinary production run
        {"name": "disk_1024x4096", "kind": "disk", "n_r": 1024, "n_phi": 4096, "order": 3,
         "limiter": True, "dtype": "f32"},
        # the largest disk of the benchmark: a high-resolution run, memory traffic
        {"name": "disk_8192x16384", "kind": "disk", "n_r": 8192, "n_phi": 16384, "order": 3,
         "limiter": True, "dtype": "f32"},
        # the default disk in double precision, as convergence studies run it
        {"name": "disk_1024x4096_f64", "kind": "disk", "n_r": 1024, "n_phi": 4096, "order": 3,
         "limiter": True, "dtype": "f64"},
        # the benchmark's batch of uneven rows: every order, linear reconstruction
        {"name": "batch_512", "kind": "rows", "n_rows": 512, "n_min": 64, "n_max": 65536,
         "orders": "234", "limiter": False, "dv": False, "entry": "step", "dtype": "f32"},
        # the same batch with its residual velocity
        {"name": "batch_512_dv", "kind": "rows", "n_rows": 512, "n_min": 64, "n_max": 65536,
         "orders": "234", "limiter": False, "dv": True, "entry": "step", "dtype": "f32"},
        # a larger batch with the paper's limited reconstructions, shifted by given amounts
        # (tracers that are only carried along)
        {"name": "batch_1000_limited", "kind": "rows", "n_rows": 1000, "n_min": 64,
         "n_max": 65536, "orders": "23", "limiter": True, "dv": False, "entry": "shift",
         "dtype": "f32"},
        # the paper's two-dimensional run at about its resolution (an odd ring length):
        # bump mesh, index function, radial sweep
        {"name": "disk2d_510x1533", "kind": "disk2d", "n_r": 510, "n_phi": 1533, "order": 2,
         "density": True, "dtype": "f32"},
        # the gradient of a disk's rollout, checkpoint-and-recompute
        {"name": "adjoint_512x2048", "kind": "adjoint", "n_r": 512, "n_phi": 2048, "order": 3,
         "limiter": False, "rows": 0, "steps": 20, "every": 10, "dtype": "f32"},
        # the gradient through the limited step on uneven rows, in double precision (a
        # limiter's branch at a near tie is decided alike there)
        {"name": "adjoint_limited_rows", "kind": "adjoint", "n_r": 0, "n_phi": 0, "order": 3,
         "limiter": True, "rows": 64, "steps": 4, "every": 4, "dtype": "f64"},
        # the fourth-order correction on a disk of point values
        {"name": "a4_512x4096", "kind": "a4", "n_r": 512, "n_phi": 4096, "order": 3,
         "limiter": True, "dtype": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(rng, n, multiple):
    """A row length near n: a multiple of `multiple` (meshes mostly are), or any."""
    return max(multiple, n // multiple * multiple) if rng.random() < 0.7 else n


def draw(rng):
    kind = rng.choice(["disk", "disk", "disk", "rows", "rows", "rows", "disk2d", "adjoint",
                       "adjoint", "a4"])
    if kind == "disk":
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        most = MAX_CELLS if dtype == "f32" else 1 << 22
        n_phi = _cells(rng, _log(rng, 128, 16384), 64)
        n_r = _log(rng, 16, max(16, min(8192, most // n_phi)))
        order = rng.choice([2, 3, 3, 3, 4])
        # the unlimited form is the linear step; order 4 is run unlimited on rings
        return {"kind": kind, "n_r": n_r, "n_phi": n_phi, "order": order,
                "limiter": order != 4 and rng.random() < 0.8, "dtype": dtype}
    if kind == "rows":
        limiter = rng.random() < 0.5
        dtype = rng.choice(["f32", "f32", "f32", "f64"])
        n_min = _log(rng, 64, 4096)
        n_max = _log(rng, n_min, 65536)
        mean = (n_max - n_min) / math.log(n_max / n_min) if n_max > n_min else n_min
        most = (8 << 20) if dtype == "f32" else (1 << 20)
        return {"kind": kind, "n_rows": _log(rng, 1, max(1, min(1000, most / mean))),
                "n_min": n_min, "n_max": n_max,
                "orders": rng.choice(["2", "3", "23"] if limiter else ["3", "4", "234"]),
                "limiter": limiter, "dv": rng.random() < 0.5,
                "entry": rng.choice(["step", "step", "shift"]), "dtype": dtype}
    if kind == "disk2d":
        dtype = rng.choice(["f32", "f32", "f64"])
        n_phi = _log(rng, 256, 2048)
        return {"kind": kind, "n_r": _log(rng, 32, 1024 if dtype == "f32" else 256),
                "n_phi": n_phi, "order": rng.choice([2, 3]), "density": rng.random() < 0.7,
                "dtype": dtype}
    if kind == "adjoint":
        dtype = rng.choice(["f32", "f32", "f64"])
        steps = rng.randint(2, 20 if dtype == "f32" else 4)
        if rng.random() < 0.5:
            return {"kind": kind, "n_r": _log(rng, 32, 512),
                    "n_phi": _cells(rng, _log(rng, 256, 2048), 64),
                    "order": rng.choice([2, 3, 4]), "limiter": False, "rows": 0, "steps": steps,
                    "every": rng.randint(2, 10), "dtype": dtype}
        # through the limiters in double precision, as listed
        limiter = dtype == "f64" and rng.random() < 0.7
        return {"kind": kind, "n_r": 0, "n_phi": 0,
                "order": rng.choice([2, 3] if dtype == "f64" else [2, 3, 4]), "limiter": limiter,
                "rows": _log(rng, 1, 64), "steps": min(steps, 4), "every": rng.randint(2, 4),
                "dtype": dtype}
    dtype = rng.choice(["f32", "f32", "f64"])
    return {"kind": "a4", "n_r": _log(rng, 16, 1024 if dtype == "f32" else 256),
            "n_phi": _cells(rng, _log(rng, 128, 4096), 64), "order": 3,
            "limiter": rng.random() < 0.8, "dtype": dtype}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _row_lengths(n_rows, n_min, n_max):
    """Log-uniform lengths (the benchmark's recipe); they belong to the case, not the seed."""
    rng = np.random.default_rng(6)
    return np.round(np.exp(rng.uniform(math.log(n_min), math.log(n_max), n_rows))).astype(np.int64)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(gen, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64)


def _disk_inputs(c, seed):
    """Rings log-spaced in [0.4, 2.5]; Sigma = r^-1/2 with a vortex at r = 1 and spiral
    modes; v0 the Keplerian rate; dv 1% of it, random at every interface; dt moves the
    inner ring by 150 cells; sub-steps per ring keep the residual Courant number below 1/2.
    The gradient's disk (limiter off, donor) takes the step of the 4096-cell disk."""
    n_r, n_phi, dtype = c["n_r"], c["n_phi"], DTYPES[c["dtype"]]
    gen = _gen(seed)
    r = 0.4 * (2.5 / 0.4) ** ((torch.arange(n_r, device=DEV, dtype=torch.float64) + 0.5) / n_r)
    omega = r ** -1.5
    cells = 75.0 * n_phi / 2048 if c["kind"] == "adjoint" else 150.0
    dphi = 2.0 * math.pi / n_phi
    dt = cells * dphi * 0.4 ** 1.5
    phi = (torch.arange(n_phi, device=DEV, dtype=torch.float64) + 0.5) * dphi
    amp, phase = _uniform(gen, 0.005, 0.02, 4), _uniform(gen, 0.0, 2.0 * math.pi, 4)
    vortex = 0.1 * torch.exp(-(r - 1.0) ** 2 / (2 * 0.05 ** 2))
    q = torch.empty((n_r, n_phi), device=DEV, dtype=dtype)
    dv = torch.empty((n_r, n_phi), device=DEV, dtype=dtype)
    nsub = torch.empty(n_r, device=DEV, dtype=torch.int32)
    rows = max(1, (1 << 23) // n_phi)
    for a in range(0, n_r, rows):  # a few rings at a time: the FP64 temporaries stay small
        rr = r[a:a + rows, None]
        f = 1.0 + vortex[a:a + rows, None] * torch.exp(-(phi - math.pi) ** 2 / (2 * 0.3 ** 2))
        for m in range(4):
            f = f + amp[m] * torch.sin((m + 1) * phi + phase[m] + 6.0 * torch.log(rr))
        q[a:a + rows] = rr ** -0.5 * f
        d = 0.01 * rr ** -1.5 * _uniform(gen, -1.0, 1.0, rr.shape[0], n_phi)
        dv[a:a + rows] = d
        nsub[a:a + rows] = torch.ceil(d.abs().amax(1) * dt / dphi / 0.5).clamp(1, 8).int()
    return {"x": workloads.uniform_nodes(n_phi, 0.0, 2.0 * math.pi), "q": q.view(-1),
            "dv": dv.view(-1), "v0": omega, "dt": dt, "nsub": nsub,
            "offset": np.arange(n_r + 1, dtype=np.int64) * n_phi,
            "order": np.full(n_r, c["order"], dtype=np.int8)}


def _rows_inputs(c, seed):
    """Rows of length 1 with widths log-uniform in [1/2, 2] x mean, 1 + three Gaussians and
    a ripple, shifts of 0.3 to 200 mean cells, dv = 0.3 dx_min sin(2 pi (3 x + phase)) / dt
    (Courant number below 0.3); a line is moved by 40.7 mean cells."""
    dtype = DTYPES[c["dtype"]]
    lens = _row_lengths(c["n_rows"], c["n_min"], c["n_max"])
    offset = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    rng = np.random.default_rng(seed)
    nodes = np.empty(int(offset[-1]) + lens.size)
    dxmin = np.empty(lens.size)
    for k, n in enumerate(lens):
        w = np.exp(rng.uniform(-math.log(2.0), math.log(2.0), n))
        x = np.concatenate([[0.0], np.cumsum(w)])
        x /= x[-1]
        nodes[offset[k] + k:offset[k + 1] + k + 1] = x
        dxmin[k] = w.min() / w.sum()
    cells = np.exp(rng.uniform(math.log(0.3), math.log(200.0), lens.size))
    if lens.size == 1:
        cells[:] = 40.7
    v0 = cells / lens
    row = torch.repeat_interleave(torch.arange(lens.size, device=DEV),
                                  torch.tensor(lens, device=DEV))
    keep = torch.tensor(np.delete(nodes, offset[1:] + np.arange(lens.size)), device=DEV)
    q = torch.ones_like(keep)
    for _ in range(3):
        centre = torch.tensor(rng.uniform(0.0, 1.0, lens.size), device=DEV)[row]
        width = torch.tensor(rng.uniform(0.02, 0.1, lens.size), device=DEV)[row]
        d = torch.remainder(keep - centre + 0.5, 1.0) - 0.5
        q += torch.exp(-d * d / (2.0 * width * width))
    phase = torch.tensor(rng.uniform(0.0, 1.0, lens.size), device=DEV)[row]
    q += 0.05 * torch.sin(2.0 * math.pi * (7.0 * keep + phase))
    dv = torch.tensor(0.3 * dxmin, device=DEV)[row] * torch.sin(2.0 * math.pi * (3.0 * keep + phase))
    orders = np.array([int(o) for o in c["orders"]], dtype=np.int8)
    return {"x": nodes, "q": q.to(dtype), "dv": dv.to(dtype) if c["dv"] else None,
            "v0": torch.tensor(v0, device=DEV), "dt": 1.0,
            "nsub": torch.ones(lens.size, device=DEV, dtype=torch.int32), "offset": offset,
            "order": np.random.default_rng(10).choice(orders, size=lens.size)}


def _disk2d_inputs(c, seed):
    w = workloads.polar_disk_2d(c["n_r"], c["n_phi"], seed=int(seed), order=c["order"])
    dtype = DTYPES[c["dtype"]]

    def put(a, t=dtype):
        return torch.tensor(a, device=DEV, dtype=t).reshape(-1).contiguous()

    # spiral modes of 1% (the workload's rings are flat away from the vortex)
    rng = np.random.default_rng(seed)
    pc, rc = 0.5 * (w.phi[1:] + w.phi[:-1]), 0.5 * (w.rf[1:] + w.rf[:-1])
    wave = 0.01 * np.sin(3.0 * pc[None, :] + 6.0 * np.log(rc)[:, None] + rng.uniform(0.0, 6.0))
    return {"x": w.phi, "q": put(w.q0 * (1.0 + wave)), "dv": put(w.dvphi), "vr": put(w.vr),
            "rf": put(w.rf, torch.float64), "v0": put(w.omega, torch.float64), "dt": w.dt,
            "nsub": put(w.nsub, torch.int32),
            "offset": np.arange(w.n_r + 1, dtype=np.int64) * w.n_phi}


def _adjoint_inputs(c, seed):
    if c["rows"]:
        d = _rows_inputs({"n_rows": c["rows"], "n_min": 64, "n_max": 65536, "dv": True,
                          "orders": str(c["order"]), "dtype": c["dtype"]}, seed)
    else:
        d = _disk_inputs(c, seed)
    noise = torch.randn(d["q"].numel(), generator=_gen(seed + 1), device=DEV, dtype=torch.float64)
    d["target"] = (d["q"].double() * (1.0 + 0.05 * noise)).to(d["q"].dtype)
    return d


def _inputs(c, seed):
    return {"disk": _disk_inputs, "a4": _disk_inputs, "rows": _rows_inputs,
            "disk2d": _disk2d_inputs, "adjoint": _adjoint_inputs}[c["kind"]](c, seed)


def prepare(case, seed):
    c, d = case, _inputs(case, seed)
    d["case"] = c
    shared = c["kind"] in ("disk", "a4", "disk2d") or (c["kind"] == "adjoint" and not c["rows"])
    order = c["order"] if c["kind"] == "disk2d" else d["order"]
    d["plan"] = ram.Plan(d["offset"], d["x"], order=order, limiter=c.get("limiter", True),
                         shared_mesh=shared, adjoint=c["kind"] == "adjoint" and c["rows"] > 0,
                         a4=c["kind"] == "a4")
    if c.get("density"):
        d["plan"].set_density([(-math.pi, math.pi, 0.1387, 0.2773, 15.0)])
    if c["kind"] == "adjoint":
        d["q"].requires_grad_(True)
        d["dv"].requires_grad_(True)
    else:
        d["out"] = torch.empty_like(d["q"])
    if c["kind"] == "disk2d":
        d["scratch"] = torch.empty_like(d["q"])
    if c.get("entry") == "shift":
        d["shift"] = d["v0"] * d["dt"]
    return d


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def run(state):
    s = state
    kind = s["case"]["kind"]
    if kind == "adjoint":
        q = autograd.rollout(s["plan"], s["q"], s["v0"], s["dt"], s["case"]["steps"], dv=s["dv"],
                             nsub=s["nsub"], checkpoint_every=s["case"]["every"])
        loss = (q - s["target"]).square().sum()
        g_q, g_dv = torch.autograd.grad(loss, (s["q"], s["dv"]))
        return {"q": q.detach(), "g_q": g_q, "g_dv": g_dv}
    if kind == "disk2d":
        ram.step_2d(s["plan"], s["q"], s["out"], s["v0"], s["dt"], s["rf"], s["vr"],
                    dvphi=s["dv"], scheme=ram.VANLEER, nsub=s["nsub"], scratch=s["scratch"])
    elif s["case"].get("entry") == "shift":
        ram.shift(s["plan"], s["q"], s["out"], s["shift"])
    else:
        ram.step(s["plan"], s["q"], s["out"], s["v0"], s["dt"], dv=s["dv"], scheme=ram.VANLEER,
                 nsub=s["nsub"])
    return s["out"]


def work(case):
    """Each field, mesh and velocity read once, each result written once; arithmetic per
    cell of the reconstruction with its partial integrals (order 2, 3, 4: about 20, 45 and
    50 operations, twice that on a non-uniform mesh, whose weights are formed from the
    widths) and about 18 per residual sub-step."""
    c = case
    e = 4 if c["dtype"] == "f32" else 8
    per = {2: 20, 3: 45, 4: 50}
    if c["kind"] in ("disk", "a4"):
        n = c["n_r"] * c["n_phi"]
        return {"bytes": 3 * e * n, "flops": n * (per[c["order"]] + 28 + (8 if c["kind"] == "a4" else 0))}
    if c["kind"] == "disk2d":
        n = c["n_r"] * c["n_phi"]
        return {"bytes": 4 * e * n, "flops": n * (2 * per[c["order"]] + 18 + 22)}
    if c["kind"] == "rows":
        n = int(_row_lengths(c["n_rows"], c["n_min"], c["n_max"]).sum())
        dv = c["dv"] and c["entry"] == "step"
        mean = sum(per[int(o)] for o in c["orders"]) / len(c["orders"])
        return {"bytes": n * (2 * e + 8 + (e if dv else 0)), "flops": n * (2 * mean + (18 if dv else 0))}
    n = int(_row_lengths(c["rows"], 64, 65536).sum()) if c["rows"] else c["n_r"] * c["n_phi"]
    one = (2 if c["rows"] else 1) * per[c["order"]] + 12
    # forward, recomputed forward, and the transpose at about twice a step's arithmetic
    return {"bytes": n * (6 * e + (8 if c["rows"] else 0)), "flops": n * 4 * one * c["steps"]}


# --------------------------------------------------------------------------
# the same in plain FP64 torch
# --------------------------------------------------------------------------

def _left(a):
    return torch.roll(a, 1, -1)


def _right(a):
    return torch.roll(a, -1, -1)


def _safe_div(num, den, ok):
    return torch.where(ok, num / torch.where(ok, den, torch.ones_like(den)), torch.zeros_like(num))


def _van_leer(q, h):
    """Harmonic mean of the one-sided slopes over centre spacings, zero at an extremum."""
    dl = (q - _left(q)) / (0.5 * (_left(h) + h))
    dr = (_right(q) - q) / (0.5 * (h + _right(h)))
    return _safe_div(2.0 * dl * dr, dl + dr, dl * dr > 0)


def _ppm(q, h, limiter):
    hm, hp = _left(h), _right(h)
    up, dn = _right(q) - q, q - _left(q)
    d = h / (hm + h + hp) * ((2 * hm + h) / (h + hp) * up + (h + 2 * hp) / (hm + h) * dn)
    if limiter:
        m = torch.minimum(d.abs(), 2 * torch.minimum(up.abs(), dn.abs()))
        d = torch.where(up * dn > 0, torch.sign(d) * m, torch.zeros_like(d))
    h2 = _right(hp)  # the face between a cell and the next
    w1 = 2 * hp * h / (h + hp) * ((hm + h) / (2 * h + hp) - (h2 + hp) / (2 * hp + h))
    w2 = -h * (hm + h) / (2 * h + hp)
    w3 = hp * (hp + h2) / (h + 2 * hp)
    R = q + h / (h + hp) * up + (w1 * up + w2 * _right(d) + w3 * d) / (hm + h + hp + h2)
    L = _left(R)
    if limiter:
        flat = (R - q) * (q - L) <= 0
        dd, qa = R - L, q - 0.5 * (L + R)
        low = ~flat & (dd * qa > dd * dd / 6)
        high = ~flat & ~low & (-dd * dd / 6 > dd * qa)
        L, R = (torch.where(flat, q, torch.where(low, 3 * q - 2 * R, L)),
                torch.where(flat, q, torch.where(high, 3 * q - 2 * L, R)))
    return L, R


def _partial(q, h, p, xi, order, limiter):
    """Integral of each edge's source cell p from its left node to the fraction xi."""
    hp, qp = h[p], torch.gather(q, 1, p)
    if order == 2:
        if limiter:
            s = _van_leer(q, h)
        else:
            s = (_right(q) - _left(q)) / (0.5 * (_left(h) + 2 * h + _right(h)))
        return hp * (qp * xi + 0.5 * torch.gather(s, 1, p) * hp * (xi * xi - xi))
    if order == 3:
        L, R = _ppm(q, h, limiter)
        L, R = torch.gather(L, 1, p), torch.gather(R, 1, p)
        six = 6 * qp - 3 * (L + R)
        return hp * (L * xi + 0.5 * (R - L + six) * xi ** 2 - six * xi ** 3 / 3)
    # mean of the two quartics through the cumulative mass at five nodes
    n = h.numel()
    cell = [torch.remainder(p + k, n) for k in range(-2, 3)]
    w = [h[k] for k in cell]
    m = [h[k] * torch.gather(q, 1, k) for k in cell]
    zero = torch.zeros_like(hp)
    z = [-(w[0] + w[1]), -w[1], zero, w[2], w[2] + w[3], w[2] + w[3] + w[4]]
    v = [-(m[0] + m[1]), -m[1], zero, m[2], m[2] + m[3], m[2] + m[3] + m[4]]
    y, total = xi * hp, zero
    for side in (0, 1):
        for k in range(side, side + 5):
            term = v[k]
            for j in range(side, side + 5):
                if j != k:
                    term = term * (y - z[j]) / (z[k] - z[j])
            total = total + 0.5 * term
    return total


def _shift64(x, q, s, order, limiter):
    """q (rows, cells) on the nodes x moved by s (rows): the cumulative mass at the shifted
    nodes, differenced and divided by the widths."""
    n, h, length = x.numel() - 1, x[1:] - x[:-1], x[-1] - x[0]
    y = x[None, :] - s[:, None]
    turns = torch.floor((y - x[0]) / length)
    y = (y - turns * length).contiguous()
    p = (torch.searchsorted(x, y, right=True) - 1).clamp(0, n - 1)
    mass = q * h
    cum = torch.cumsum(mass, 1)
    before = torch.gather(cum - mass, 1, p)
    at = turns * cum[:, -1:] + before + _partial(q, h, p, (y - x[p]) / h[p], order, limiter)
    return (at[:, 1:] - at[:, :-1]) / h


def _residual64(x, q, dv, dt, nsub, scheme):
    h = x[1:] - x[:-1]
    for k in range(int(nsub.max())):
        c = dv * (dt / nsub.double())[:, None]
        if scheme == ram.VANLEER:
            half = 0.5 * _van_leer(q, h.expand_as(q))
            from_left, from_right = _left(q + half * h) - _left(half) * c, q - half * (h + c)
        else:
            from_left, from_right = _left(q), q
        flux = c * torch.where(c > 0, from_left, from_right)
        q = torch.where((k < nsub)[:, None], q - (_right(flux) - flux) / h, q)
    return q


def _radial64(rf, q, vr, dt):
    width, centre = (rf[1:] - rf[:-1])[:, None], 0.5 * (rf[1:] + rf[:-1])[:, None]
    slope = torch.zeros_like(q)
    grad = (q[1:] - q[:-1]) / (centre[1:] - centre[:-1])
    dl, dr = grad[:-1], grad[1:]
    slope[1:-1] = _safe_div(2.0 * dl * dr, dl + dr, dl * dr > 0)
    v = vr[1:-1]
    low = q[:-1] + 0.5 * slope[:-1] * (width[:-1] - v * dt)
    high = q[1:] - 0.5 * slope[1:] * (width[1:] + v * dt)
    flux = torch.zeros_like(vr)
    flux[1:-1] = rf[1:-1, None] * v * torch.where(v > 0, low, high)
    area = 0.5 * (rf[1:] ** 2 - rf[:-1] ** 2)[:, None]
    return q - dt * (flux[1:] - flux[:-1]) / area


def _a4_divide(q, inverse):
    """The circulant (1, 22, 1) / 24, or its inverse, by its spectrum."""
    n = q.shape[1]
    k = torch.arange(n // 2 + 1, device=q.device, dtype=torch.float64)
    eig = (22.0 + 2.0 * torch.cos(2.0 * math.pi * k / n)) / 24.0
    f = torch.fft.rfft(q, dim=1)
    return torch.fft.irfft(f / eig if inverse else f * eig, n=n, dim=1)


def _blocks(d):
    """Row ranges that one 2D tensor holds: rows of one mesh a few at a time, own meshes
    one by one.  Yields (first row, last row + 1, nodes on the device)."""
    offset, x = d["offset"], d["x"]
    n_rows = offset.size - 1
    shared = x.size == offset[1] + 1 and n_rows > 1 or n_rows == 1
    if shared:
        xs = torch.tensor(x, device=DEV)
        step = max(1, (1 << 21) // int(offset[1]))
        for a in range(0, n_rows, step):
            yield a, min(n_rows, a + step), xs
    else:
        for r in range(n_rows):
            yield r, r + 1, torch.tensor(x[offset[r] + r:offset[r + 1] + r + 1], device=DEV)


def _step64(c, d, q, dv, scheme, steps=1, out_like=None):
    """`steps` steps of the packed field q (FP64), block by block."""
    parts = []
    for a, b, x in _blocks(d):
        lo, hi, n = int(d["offset"][a]), int(d["offset"][b]), x.numel() - 1
        f = q[lo:hi].view(b - a, n)
        v = None if dv is None else dv[lo:hi].view(b - a, n)
        order = c["order"] if c["kind"] == "disk2d" else int(d["order"][a])
        for _ in range(steps):
            if c["kind"] == "a4":
                f = _a4_divide(f, False)
            f = _shift64(x, f, d["v0"][a:b] * d["dt"], order, c.get("limiter", True))
            if c["kind"] == "a4":
                f = _a4_divide(f, True)
            if v is not None:
                f = _residual64(x, f, v, d["dt"], d["nsub"][a:b], scheme)
        parts.append(f.reshape(-1))
    return torch.cat(parts)


def exact(case, seed):
    c, d = case, _inputs(case, seed)
    q = d["q"].double()
    dv = None if d["dv"] is None or c.get("entry") == "shift" else d["dv"].double()
    if c["kind"] == "adjoint":
        q.requires_grad_(True)
        dv.requires_grad_(True)
        end = _step64(c, d, q, dv, ram.DONOR, c["steps"])
        loss = (end - d["target"].double()).square().sum()
        g_q, g_dv = torch.autograd.grad(loss, (q, dv))
        return {"q": end.detach(), "g_q": g_q, "g_dv": g_dv}
    out = _step64(c, d, q, dv, ram.VANLEER)
    if c["kind"] == "disk2d":
        n_r, n_phi = c["n_r"], c["n_phi"]
        out = _radial64(d["rf"], out.view(n_r, n_phi), d["vr"].double().view(n_r + 1, n_phi),
                        d["dt"]).reshape(-1)
    return out
