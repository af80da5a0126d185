"""The work a user of this package has it do, as cases that can be timed and compared.

Three kinds of case, each one pass through the public Python API:

- ``solve``: a periodic or walled grid is initialised from theta0 and its
  gradient (or theta0 alone), advanced a number of steps and recovered
  (``Solver.set_theta0``, ``step``, ``macros``; with ``norms`` also
  ``sum_theta`` and ``reduce`` against reference data);
- ``batch``: many independent 2D grids advanced together (``Batch``);
- ``gradient``: one training step through ``burgers_fields``: forward to
  u(T), theta(T), a data misfit, and its gradients to theta0 and nu.

Initial fields are 1.5 plus a few Fourier modes (cosines across an axis with
walls), or Example 1's exp(a cos(pi x) / (2 pi nu)), made from the seed.
``exact`` runs the scheme as the paper states it (collision with the dense
q x q matrix, streaming by rolls, walls by even reflection onto the doubled
periodic grid) in 64-bit torch.
"""

from __future__ import annotations

import itertools
import math

import torch

from paper_2309_02825_gb300 import lb
from paper_2309_02825_gb300.adjoint import burgers_fields

DEV = "cuda"


def listed():
    return [
        # Example 1 of the paper (walls at x = 0 and 1, one refinement): the
        # smallest grid, many steps: launches and latency
        {"name": "walls_1d_81", "kind": "solve", "d": 1, "n0": 81, "steps": 800, "eps": 1.0, "precision": "fp64",
         "walls": 1, "start": "example1"},
        # a smoke-sized 2D solve in the default precision: the shortest call
        {"name": "solve_2d_64", "kind": "solve", "d": 2, "n0": 64, "n1": 64, "steps": 20, "eps": 0.2048,
         "precision": "fp64", "grad": True},
        # a mid-size convergence run of the 2D family whose state stays in L2
        {"name": "solve_2d_512", "kind": "solve", "d": 2, "n0": 512, "n1": 512, "steps": 128, "eps": 0.2048,
         "precision": "fx64", "grad": True, "norms": True},
        # the benchmark's headline: 4096^2 fixed point, schedule picked once by
        # autotune, initialise + 100 sweeps + recovery + total + norms
        {"name": "solve_2d_4096", "kind": "solve", "d": 2, "n0": 4096, "n1": 4096, "steps": 100, "eps": 0.2048,
         "precision": "fx64", "grad": True, "norms": True, "autotune": True},
        # a ragged grid in FP32-shifted storage, theta0 only, no tuning
        {"name": "solve_2d_1999x1501", "kind": "solve", "d": 2, "n0": 1999, "n1": 1501, "steps": 100, "eps": 0.2048,
         "precision": "fp32s", "grad": False},
        # a large grid in the default precision and schedule
        {"name": "solve_2d_2048", "kind": "solve", "d": 2, "n0": 2048, "n1": 2048, "steps": 40, "eps": 0.2048,
         "precision": "fp64", "grad": True},
        # the 3D family at its largest size, fixed point
        {"name": "solve_3d_256", "kind": "solve", "d": 3, "n0": 256, "n1": 256, "n2": 256, "steps": 32, "eps": 0.0512,
         "precision": "fx64", "grad": True},
        # a small ragged 3D grid in FP32-shifted storage
        {"name": "solve_3d_101x90x77", "kind": "solve", "d": 3, "n0": 101, "n1": 90, "n2": 77, "steps": 33,
         "eps": 0.0512, "precision": "fp32s", "grad": True, "norms": True},
        # Example 4 of the paper at its finest printed level
        {"name": "solve_4d_50", "kind": "solve", "d": 4, "n0": 50, "n1": 50, "n2": 50, "n3": 50, "steps": 10,
         "eps": 0.08, "precision": "fx64", "grad": True},
        # batched instances of mixed sizes (log-uniform 32 .. 512), tuned once
        {"name": "batch_64", "kind": "batch", "count": 64, "lo": 32, "hi": 512, "steps": 200, "precision": "fp32s",
         "autotune": True},
        # the adjoint family's training step (fixed point, gradients to theta0 and nu)
        {"name": "gradient_2d_512", "kind": "gradient", "d": 2, "n0": 512, "n1": 512, "steps": 256, "eps": 0.2048,
         "precision": "fx64"},
        # a small training step in the default precision
        {"name": "gradient_2d_160x128", "kind": "gradient", "d": 2, "n0": 160, "n1": 128, "steps": 100, "eps": 0.2048,
         "precision": "fp64"},
    ]


_EPS = {1: 0.16, 2: 0.2048, 3: 0.0512, 4: 0.08}


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def sizes(d, nodes):
        # a box of about `nodes` nodes, each axis within a factor 1.5 of the cube's edge
        edge = nodes ** (1.0 / d)
        return {"n%d" % a: max(4, int(round(edge * rng.uniform(0.67, 1.5)))) for a in range(d)}

    def steps(d, c, most):
        # at most the diffusion time at which the lowest mode has lost about half
        # of its amplitude, so that u keeps its size
        n = min(c["n%d" % a] for a in range(d))
        return logint(4, max(5, min(most, int(n * n / (64.0 * c["eps"])))))

    what = rng.random()
    precision = rng.choice(["fp64", "fx64", "fp32s"])
    if what < 0.12:
        return {"kind": "batch", "count": logint(8, 128), "lo": 32, "hi": rng.choice([128, 256, 512]),
                "steps": logint(16, 256), "precision": rng.choice(["fp32s", "fx64"]), "autotune": rng.random() < 0.5}
    if what < 0.3:
        d = rng.choice([1, 2, 2, 2, 3])
        c = {"kind": "gradient", "d": d, "eps": _EPS[d] * rng.uniform(0.7, 1.3), "precision": precision}
        c.update(sizes(d, {1: logint(32, 512), 2: logint(2000, 262144), 3: logint(4000, 110000)}[d]))
        c["steps"] = steps(d, c, 200)
        return c
    d = rng.choice([1, 2, 2, 2, 2, 3, 3, 4])
    c = {"kind": "solve", "d": d, "eps": _EPS[d] * rng.uniform(0.7, 1.3), "precision": precision,
         "grad": rng.random() < 0.7, "norms": rng.random() < 0.4}
    nodes = {1: logint(16, 1000), 2: logint(1000, 12000000), 3: logint(4000, 12000000), 4: logint(10000, 4000000)}[d]
    c.update(sizes(d, nodes))
    most = {1: 2000, 2: 100, 3: 32, 4: 10}[d]
    c["steps"] = steps(d, c, most)
    if d <= 3 and rng.random() < 0.25:
        c["walls"] = rng.randrange(1, 1 << d)  # bit a: walls at both ends of axis a
    elif d == 2 and rng.random() < 0.4:
        c["autotune"] = True
    return c


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------

def _axes(c):
    return [c["n%d" % a] for a in range(c["d"])]


def _units(c):
    """(N, nu, dx, dt, mirror axes): unit length along x, eps = nu dt / dx^2."""
    N = _axes(c)
    walls = int(c.get("walls", 0) or 0)
    dx = 1.0 / (N[0] - 1 if walls & 1 else N[0])
    if c.get("start") == "example1":
        dt = 16.0 * dx * dx  # Example 1: dx = 1/40 / 2^l, dt = 1/100 / 4^l
        return N, c["eps"] * dx * dx / dt, dx, dt, walls
    nu = {1: 0.05, 2: 0.02, 3: 0.01, 4: 0.1}[c["d"]]
    return N, nu, dx, c["eps"] * dx * dx / nu, walls


def _field(N, dx, walls, modes, offset):
    """(theta, grad theta) of offset + sum_m amp_m prod_a (wave of axis a), on the GPU."""
    d = len(N)
    shape = tuple(reversed(N))
    th = torch.full(shape, offset, dtype=torch.float64, device=DEV)
    gr = torch.zeros((d,) + shape, dtype=torch.float64, device=DEV)
    for k, amp, phase in modes:
        waves, slopes = [], []
        for a in range(d):
            x = torch.arange(N[a], dtype=torch.float64, device=DEV) * dx
            view = [1] * d
            view[d - 1 - a] = N[a]
            if (walls >> a) & 1:
                w = math.pi * k[a] / ((N[a] - 1) * dx)
                f, g = torch.cos(w * x).to(torch.complex128), (-w * torch.sin(w * x)).to(torch.complex128)
                g[0] = 0
                g[-1] = 0
            else:
                w = 2.0 * math.pi * k[a] / (N[a] * dx)
                f = torch.polar(torch.ones_like(x), w * x)
                g = 1j * w * f
            waves.append(f.reshape(view))
            slopes.append(g.reshape(view))
        rot = amp * complex(math.cos(phase), math.sin(phase))
        for a in range(-1, d):
            prod = rot
            for b in range(d):
                prod = prod * (slopes[b] if a == b else waves[b])
            (th if a < 0 else gr[a]).add_(prod.real)
    return th, gr


def _modes(d, count, seed):
    """Seeded modes 0 < |k| <= 3 with small amplitudes (theta stays above 0.5)."""
    g = torch.Generator().manual_seed(int(seed))
    ks = [v for v in itertools.product(range(-2, 3), repeat=d) if 0 < sum(x * x for x in v) <= 9]
    pick = torch.randint(0, len(ks), (count,), generator=g).tolist()
    amp = (0.03 + 0.1 * torch.rand(count, generator=g, dtype=torch.float64)).tolist()
    phase = (2.0 * math.pi * torch.rand(count, generator=g, dtype=torch.float64)).tolist()
    return [(ks[i], a, p) for i, a, p in zip(pick, amp, phase)]


def _start(c, seed):
    N, nu, dx, dt, walls = _units(c)
    if c.get("start") == "example1":
        g = torch.Generator().manual_seed(int(seed))
        amp = 0.5 + 0.5 * float(torch.rand(1, generator=g, dtype=torch.float64))
        x = torch.arange(N[0], dtype=torch.float64, device=DEV) * dx
        th = torch.exp(amp * torch.cos(math.pi * x) / (2.0 * math.pi * nu))
        gr = (-amp * torch.sin(math.pi * x) / (2.0 * nu) * th)
        gr[0] = 0
        gr[-1] = 0
        return th, gr[None].contiguous()
    return _field(N, dx, walls, _modes(c["d"], 6, seed), 1.5)


def _reference(c, seed):
    """Reference data of the norms and the misfit: the initial fields of slightly
    other modes with 1e-3 of noise, as measured data has."""
    N, nu, dx, dt, walls = _units(c)
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 77)
    th, gr = _field(N, dx, walls, [(k, 0.9 * a, p) for k, a, p in _modes(c["d"], 6, seed)], 1.5)
    th += 1e-3 * torch.randn(th.shape, generator=g, dtype=torch.float64, device=DEV)
    u = -2.0 * nu * gr / th
    return th, u


def _batch(c, seed):
    g = torch.Generator().manual_seed(20 + c["count"])  # the sizes belong to the case, the fields to the seed
    lo, hi = math.log(c["lo"]), math.log(c["hi"])
    n = torch.exp(lo + (hi - lo) * torch.rand(2 * c["count"], generator=g, dtype=torch.float64)).round().int().tolist()
    nu = torch.exp(math.log(0.005) + math.log(20.0) * torch.rand(c["count"], generator=g, dtype=torch.float64)).tolist()
    sizes = [(n[2 * j], n[2 * j] if j % 4 else n[2 * j + 1]) for j in range(c["count"])]  # one in four is not square
    dx = [1.0 / s[0] for s in sizes]
    dt = [4.0 * h * h for h in dx]
    th, gr = zip(*(_field(s, h, 0, _modes(2, 3, 7919 * int(seed) + j), 1.5) for j, (s, h) in enumerate(zip(sizes, dx))))
    return sizes, nu, dx, dt, th, gr


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        sizes, nu, dx, dt, th, gr = _batch(c, seed)
        b = lb.Batch(sizes, nu, dx, dt, precision=c["precision"],
                     theta_ref=[1.5] * len(sizes) if c["precision"] == "fp32s" else None)
        if c.get("autotune"):
            b.autotune()
        flat_th = torch.cat([t.reshape(-1) for t in th])
        flat_gr = torch.cat([t.reshape(-1) for t in gr])
        return {"case": c, "batch": b, "theta0": flat_th, "grad0": flat_gr}
    N, nu, dx, dt, walls = _units(c)
    th, gr = _start(c, seed)
    state = {"case": c, "theta0": th}
    if c["kind"] == "gradient":
        state["data"] = _reference(c, seed)
        state["args"] = (c["d"], N, dx, dt, c["steps"])
        state["nu"] = nu
        return state
    ref = float(th.mean()) if c["precision"] == "fp32s" else 0.0
    state["solver"] = lb.Solver(c["d"], N, nu, dx, dt, precision=c["precision"], theta_ref=ref,
                                boundary=["mirror" if (walls >> a) & 1 else "periodic" for a in range(c["d"])]
                                if walls else None)
    if c.get("autotune"):
        state["solver"].autotune()
    state["grad0"] = gr if c.get("grad", True) else None
    if c.get("norms"):
        state["data"] = _reference(c, seed)
    return state


# ---------------------------------------------------------------------------
# One pass.
# ---------------------------------------------------------------------------

def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        b = state["batch"]
        b.set_theta0(state["theta0"], state["grad0"])
        b.step(c["steps"])
        return list(b.macros())
    if c["kind"] == "gradient":
        d, N, dx, dt, T = state["args"]
        th0 = state["theta0"].detach().requires_grad_(True)
        nu = torch.tensor(state["nu"], dtype=torch.float64, requires_grad=True)
        u, th = burgers_fields(th0, nu, d, N, dx, dt, T, precision=c["precision"])
        ref_th, ref_u = state["data"]
        loss = 0.5 * ((u - ref_u).square().mean() + (th - ref_th).square().mean())
        loss.backward()
        return {"u": u.detach(), "theta": th.detach(), "dtheta0": th0.grad, "dnu": nu.grad}
    s = state["solver"]
    s.set_theta0(state["theta0"], state["grad0"])
    s.step(c["steps"])
    th, gr, u = s.macros()
    out = {"theta": th, "grad": gr, "u": u}
    if c.get("norms"):
        norms = s.reduce(th, u, *state["data"])
        out["sum"] = s.sum_theta()
        out["norms"] = [norms["sum_theta"]] + [v for k in sorted(norms) if k != "sum_theta"
                                               for v in norms[k].values()]
    return out


# Floating-point operations of one node's collision in moment form, by d.
_OPS = {1: 9, 2: 38, 3: 92, 4: 170}


def work(case):
    c = case
    if c["kind"] == "batch":
        g = torch.Generator().manual_seed(20 + c["count"])
        lo, hi = math.log(c["lo"]), math.log(c["hi"])
        n = torch.exp(lo + (hi - lo) * torch.rand(2 * c["count"], generator=g, dtype=torch.float64)).round().int().tolist()
        nodes = sum(n[2 * j] * (n[2 * j] if j % 4 else n[2 * j + 1]) for j in range(c["count"]))
        return {"bytes": nodes * 8 * 6, "flops": nodes * c["steps"] * _OPS[2]}  # theta0, grad0; theta, u
    d = c["d"]
    nodes = math.prod(_axes(c))
    if c["kind"] == "gradient":
        # forward, and a reverse step of the transposed collision with the nu term
        return {"bytes": nodes * 8 * (1 + 2 * (d + 1) + 1), "flops": nodes * c["steps"] * 3 * _OPS[d]}
    data = (d + 1) if c.get("norms") else 0
    inputs = 1 + (d if c.get("grad", True) else 0) + data
    return {"bytes": nodes * 8 * (inputs + 1 + 2 * d), "flops": nodes * c["steps"] * _OPS[d]}


# ---------------------------------------------------------------------------
# The scheme in 64-bit torch, as the paper states it.
# ---------------------------------------------------------------------------

def _velocities(d):
    e = [[0] * d]
    for s in (1, -1):
        for a in range(d):
            v = [0] * d
            v[a] = s
            e.append(v)
    for a in range(d):
        for b in range(a + 1, d):
            for sa, sb in ((1, 1), (-1, 1), (-1, -1), (1, -1)):
                v = [0] * d
                v[a], v[b] = sa, sb
                e.append(v)
    return e


def _scheme(d, eps):
    """(velocities, M, S, w, s1, sigma): natural moments, Theorem 2's rates and
    weights; eps a 64-bit tensor (0-dim), so that autograd sees d/deps."""
    e = torch.tensor(_velocities(d), dtype=torch.float64, device=DEV)
    one = torch.ones((), dtype=torch.float64, device=DEV)
    s1 = 2.0 / (6.0 * eps + 1.0)
    s2 = 24.0 * eps / (6.0 * eps + 1.0) ** 2
    s22 = 4.0 / (6.0 * eps + 3.0)
    w1 = (one / 6.0 - (d - 1) * eps / 3.0) if d > 1 else one / 6.0
    wd = eps / 6.0 if d > 1 else 0.0 * eps
    rows, rates = [torch.ones(len(e), dtype=torch.float64, device=DEV)], [one]
    for a in range(d):
        rows.append(e[:, a])
        rates.append(s1)
    for a in range(d):
        rows.append(e[:, a] ** 2)
        rates.append(s2)
    for a in range(d):
        for b in range(a + 1, d):
            rows.append(e[:, a] * e[:, b])
            rates.append(s22)
    for a in range(d):
        for b in range(d):
            if a != b:
                rows.append(e[:, a] ** 2 * e[:, b])
                rates.append(one)
    for a in range(d):
        for b in range(a + 1, d):
            rows.append(e[:, a] ** 2 * e[:, b] ** 2)
            rates.append(one)
    w0 = 1.0 - 2 * d * w1 - 2 * d * (d - 1) * wd
    w = torch.stack([w0] + [w1] * (2 * d) + [wd] * (2 * d * (d - 1)))
    sigma = 2.0 * w1 + 4.0 * (d - 1) * wd
    return e, torch.stack(rows), torch.stack(rates), w, s1, sigma


def _advance(th0, gr0, steps, d, eps, dx, dt, reverse=False):
    """(theta, grad, u) after `steps` steps on a periodic grid, all 64-bit."""
    e, M, S, w, s1, sigma = _scheme(d, eps)
    Mi = torch.linalg.inv(M)
    q = len(e)
    shape = th0.shape
    flat = th0.reshape(1, -1)
    g = (w[:, None] * (e / dt * dx)) @ gr0.reshape(d, -1)
    f = w[:, None] * flat - dt * ((Mi @ torch.diag(1.0 / S) @ M) @ g)
    relax = Mi @ torch.diag(S) @ M
    K = torch.eye(q, dtype=torch.float64, device=DEV) - relax @ (
        torch.eye(q, dtype=torch.float64, device=DEV) - w[:, None].expand(q, q))
    ei = _velocities(d)
    dims = [d - 1 - a for a in range(d)]
    for _ in range(steps):
        f = (K @ f).reshape((q,) + tuple(shape))
        f = torch.stack([torch.roll(f[i], ei[i], dims) if any(ei[i]) else f[i] for i in range(q)]).reshape(q, -1)
    th = f.sum(0)
    J = e.T @ f
    grad = -s1 * J / (sigma * dx)
    u = (2.0 - s1) * (dx / dt) * J / th
    return th.reshape(shape), grad.reshape((d,) + tuple(shape)), u.reshape((d,) + tuple(shape))


def _central4(th, d, dx):
    g = []
    for a in range(d):
        r = lambda k: torch.roll(th, k, d - 1 - a)  # noqa: E731
        g.append((8.0 * (r(-1) - r(1)) - (r(-2) - r(2))) / (12.0 * dx))
    return torch.stack(g)


def _double(t, N, walls, odd=None):
    """Even reflection of a field across the walls (odd along axis `odd`)."""
    d = len(N)
    for a in range(d):
        if (walls >> a) & 1:
            dim = d - 1 - a
            back = t.narrow(dim, 1, N[a] - 2).flip(dim)
            t = torch.cat([t, -back if odd == a else back], dim)
    return t


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        sizes, nu, dx, dt, th, gr = _batch(c, seed)
        out_t, out_u = [], []
        for j in range(len(sizes)):
            eps = torch.tensor(nu[j] * dt[j] / dx[j] ** 2, dtype=torch.float64, device=DEV)
            t, _, u = _advance(th[j], gr[j], c["steps"], 2, eps, dx[j], dt[j])
            out_t.append(t.reshape(-1))
            out_u.append(u.reshape(-1))
        return [torch.cat(out_t), torch.cat(out_u)]
    d = c["d"]
    N, nu, dx, dt, walls = _units(c)
    th0, gr0 = _start(c, seed)
    if c["kind"] == "gradient":
        if math.prod(N) * (1 + 2 * d * d) * 8 * 4 * c["steps"] > 60e9:
            return None
        th0 = th0.requires_grad_(True)
        nu_t = torch.tensor(nu, dtype=torch.float64, device=DEV, requires_grad=True)
        t, _, u = _advance(th0, _central4(th0, d, dx), c["steps"], d, nu_t * dt / dx ** 2, dx, dt)
        ref_th, ref_u = _reference(c, seed)
        (0.5 * ((u - ref_u).square().mean() + (t - ref_th).square().mean())).backward()
        return {"u": u.detach(), "theta": t.detach(), "dtheta0": th0.grad, "dnu": nu_t.grad}
    if math.prod(N) * c["steps"] * (1 + 2 * d * d) ** 2 > 2e11:
        return None
    eps = torch.tensor(nu * dt / dx ** 2, dtype=torch.float64, device=DEV)
    full = _double(th0, N, walls)
    if not c.get("grad", True):
        grads = _central4(full, d, dx)
    else:
        grads = torch.stack([_double(gr0[a], N, walls, odd=a) for a in range(d)])
    for a in range(d):
        if (walls >> a) & 1:
            grads[a].select(d - 1 - a, 0).zero_()
            grads[a].select(d - 1 - a, N[a] - 1).zero_()
    t, g, u = _advance(full, grads, c["steps"], d, eps, dx, dt)
    cut = tuple(slice(0, n) for n in reversed(N))
    t, g, u = t[cut], g[(slice(None),) + cut], u[(slice(None),) + cut]
    out = {"theta": t, "grad": g, "u": u}
    if c.get("norms"):
        weight = torch.ones_like(t)
        for a in range(d):
            if (walls >> a) & 1:
                weight.select(d - 1 - a, 0).mul_(0.5)
                weight.select(d - 1 - a, N[a] - 1).mul_(0.5)
        out["sum"] = float((weight * t).sum())
        ref_th, ref_u = _reference(c, seed)
        norms = [float(t.sum())]
        for x, y in [(t, ref_th)] + [(u[a], ref_u[a]) for a in range(d)]:
            diff = x - y
            norms += [float(diff.square().mean().sqrt()), float(diff.abs().max()),
                      float((diff.square().sum() / y.square().sum()).sqrt())]
        out["norms"] = norms
    return out
