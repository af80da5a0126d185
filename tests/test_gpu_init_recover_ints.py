"""Single-precision initialisation and the recovery's quotient, both formed on
the integer pipes, against FP64 and IEEE division."""

import numpy as np
import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu

SHAPES = {1: (301,), 2: (67, 41), 3: (13, 11, 9), 4: (7, 6, 5, 5)}
EPS = {1: 0.16, 2: 0.2048, 3: 0.0512, 4: 0.08}


def _velocities(d):
    e = [[0] * d]
    for s in (1, -1):
        for a in range(d):
            e.append([s if b == a else 0 for b in range(d)])
    for a in range(d):
        for b in range(a + 1, d):
            for sa, sb in ((1, 1), (-1, 1), (-1, -1), (1, -1)):
                v = [0] * d
                v[a], v[b] = sa, sb
                e.append(v)
    return e


@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("case", ["run", "near the reference", "flat", "large gradient", "outside the range"])
def test_fp32_initialisation_is_rounded_once(d, case):
    """Each stored value is the exact population rounded to FP32, up to the
    formation's own rounding: constants at 2^-53 of themselves, theta and the
    gradient aligned at 2^-60 of the larger, so below 2^-48 of the terms' sum;
    beyond the aligned range of magnitudes the FP64 form, within the same."""
    N = SHAPES[d]
    shape = tuple(reversed(N))
    rng = np.random.default_rng(11 * d)
    th = 1.5 + 0.4 * rng.standard_normal(shape).clip(-3, 3)
    g = rng.standard_normal((d,) + shape)
    dx = 1.0 / N[0]
    if case == "near the reference":
        th = 1.5 + 1e-9 * rng.standard_normal(shape)
        th.flat[::5] = 1.5
    elif case == "flat":
        th.flat[::3] = 1.5
        g[:] = 0.0
    elif case == "large gradient":
        g *= 1e7
    elif case == "outside the range":  # theta - theta_ref below 2^-40, no gradient
        th = 1.5 + 2.0 ** -45 * rng.integers(-9, 9, shape)
        g *= 1e-14
    s = lb.Solver(d, N, 0.02, dx, EPS[d] * dx * dx / 0.02, precision="fp32s", theta_ref=1.5)
    s.set_theta0(torch.from_numpy(th).cuda(), torch.from_numpy(g).cuda())
    pitch, slab, eb = s.state_layout()
    p = s.params
    buf = s.save_state().cpu().numpy().view(np.float32)
    s.close()
    e = _velocities(d)
    q = len(e)
    rows = int(np.prod(N[1:]))
    got = [buf[i * slab:i * slab + rows * pitch].reshape(rows, pitch)[:, :N[0]].reshape(shape) for i in range(q)]
    sigma = p["cs2"] / p["c"] ** 2
    wd = p["wd"] if d > 1 else 0.0
    iax = 0.5 * dx * (sigma / p["s1"] - 4.0 * (d - 1.0) * wd)
    idg = wd * dx
    L = np.longdouble
    dth, gl = (th - 1.5).astype(L), g.astype(L)
    scale = np.abs(dth) + dx * np.abs(gl).sum(0)
    for i in range(q):
        ax = [a for a in range(d) if e[i][a]]
        if not ax:
            f = L(p["w0"]) * dth
        elif len(ax) == 1:
            f = L(p["w1"]) * dth - e[i][ax[0]] * L(iax) * gl[ax[0]]
        else:
            f = L(wd) * dth - L(idg) * sum(e[i][a] * gl[a] for a in ax)
        f = np.roll(f, [-v for v in reversed(e[i])], tuple(range(d)))  # stored at x - e_i
        sz = np.roll(scale, [-v for v in reversed(e[i])], tuple(range(d)))
        tol = np.abs(f) * L(2.0) ** -24 + sz * L(2.0) ** -48
        assert np.all(np.abs(got[i].astype(L) - f) <= tol), (i, float(np.max(np.abs(got[i] - f) / tol)))


def test_recovered_velocity_is_the_ieee_quotient():
    """J = 1 at every node, so u is (2 - s1) c / theta: bit for bit the division
    that IEEE 754 rounds, over powers of two, their neighbours and random values."""
    rng = np.random.default_rng(3)
    one = np.ldexp(1.0, np.arange(-1, 12))
    th = np.concatenate([one, np.nextafter(one, 0), np.nextafter(one, 1e9), 4.0 + 1e-15 * np.arange(200),
                         rng.uniform(2.1, 4.2, 60000), np.exp(rng.uniform(1.0, 9.0, 60000))])
    n = th.size
    s = lb.Solver(1, (n,), 0.05, 1.0 / n, 0.16 / n**2 / 0.05, precision="fp64")
    one_n = torch.ones(n, dtype=torch.float64, device="cuda")
    s.set_theta0(one_n, torch.zeros(1, n, dtype=torch.float64, device="cuda"))
    pitch, slab, eb = s.state_layout()
    state = np.zeros((3, slab))
    state[0, :n], state[1, :n], state[2, :n] = th - 2.0, 1.5, 0.5
    s.load_state(torch.from_numpy(state.reshape(-1)).cuda().view(torch.uint8), 0)
    got_th, _, u = s.macros(want=("theta", "u"))
    got_th, u = got_th.cpu().numpy(), u.cpu().numpy().reshape(-1)
    p = s.params
    s.close()
    ok = got_th > 0
    assert ok.sum() > 0.99 * n
    want = ((2.0 - p["s1"]) * p["c"]) / got_th
    assert np.array_equal(u[ok], want[ok])


@pytest.mark.parametrize("N", [(1,), (3,), (37,), (5, 4), (67, 41), (9, 2, 7), (6, 5, 4, 3)])
@pytest.mark.parametrize("walls", [False, True])
def test_central_difference_in_integers(N, walls):
    """The gradient that lb_set_theta0 forms is the fourth-order difference rounded
    once and multiplied by 1 / (12 dx): within 2 ulp of itself where the exponents
    of theta allow the integers, else within 8 roundings of the largest term.  Read
    off the fixed-point state's J = -(sigma dx / s1) grad, whose own rounding is
    2^-57 of max|theta| per population."""
    if walls and min(N) < 5:
        pytest.skip("walls need five nodes")
    d = len(N)
    shape = tuple(reversed(N))
    rng = np.random.default_rng(sum(N))
    th = rng.uniform(0.9, 3.0, shape)
    th.flat[::7] *= 2.0 ** rng.integers(-9, 9, th.flat[::7].shape)
    dx = 1.0 / 16
    kw = {"boundary": ["mirror"] * d} if walls else {}
    grads = []
    for given in (False, True):
        s = lb.Solver(d, N, 0.02, dx, EPS[d] * dx * dx / 0.02, precision="fx64", **kw)
        g = None
        if given:
            L = np.longdouble
            g = np.empty((d,) + shape)
            for a in range(d):
                ax, n = d - 1 - a, N[a]
                idx = np.arange(n)
                def at(m):
                    j = idx + m
                    if walls:
                        j = np.where(j < 0, -j, j)
                        j = np.where(j >= n, 2 * (n - 1) - j, j)
                    return np.take(th, j % n if not walls else j, axis=ax).astype(L)
                g[a] = ((at(-2) - at(2) + 8 * (at(1) - at(-1))) / (12 * L(dx))).astype(np.float64)
            g = torch.from_numpy(g).cuda()
        s.set_theta0(torch.from_numpy(th).cuda(), g)
        grads.append(s.macros()[1].cpu().numpy())
        s.close()
    big = np.abs(th).max()
    tol = 18 * big / (12 * dx) * 2.0 ** -49
    assert np.abs(grads[0] - grads[1]).max() <= tol
