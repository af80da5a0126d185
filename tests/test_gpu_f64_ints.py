"""The FP64 collision formed on the integer pipes against exact rational arithmetic.

One sweep over a loaded state whose nodes cover the dispatch: magnitudes like
those of a run (every exponent within the alignment width), exponents spread
wider, zeros, subnormals, sums at the 2^62 limit, mixed signs, infinities and
NaN.  Each finite result must lie within 16 roundings of the sum of the node's
magnitudes (the direct FP64 form's own bound); where all exponents lie within
the alignment width and the magnitudes' sum leaves no doubt, within one
rounding of the result plus the products' rounding.
"""

from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu

SHAPES = {2: (37, 11), 3: (13, 6, 5), 4: (9, 5, 4, 3)}
WIDTH = {2: 7, 3: 5, 4: 5}


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


def _collide_exact(f, d, p):
    """Closed-form collision in rationals; f a list of q Fractions."""
    e = _velocities(d)
    s2, s22, wd, sigma = (Fraction(p[k]) for k in ("s2x", "s22", "wd", "sigma"))
    k1, k2, k3 = (1 - Fraction(p["s1"])) / 2, (1 - s2) / 2, (1 - s22) / 4
    cA = s2 * sigma / 2 - 2 * (d - 1) * wd
    th = sum(f)
    J = [sum(e[i][a] * f[i] for i in range(len(f))) for a in range(d)]
    P = [sum(e[i][a] ** 2 * f[i] for i in range(len(f))) for a in range(d)]
    out = [None] * len(f)
    for i in range(1, len(f)):
        ax = [a for a in range(d) if e[i][a]]
        if len(ax) == 1:
            a = ax[0]
            out[i] = k2 * P[a] + cA * th + e[i][a] * k1 * J[a]
        else:
            a, b = ax
            Pab = sum(e[j][a] * e[j][b] * f[j] for j in range(len(f)))
            out[i] = wd * th + e[i][a] * e[i][b] * k3 * Pab
    out[0] = th - sum(out[1:])
    return out


@pytest.mark.parametrize("kind", ["run", "spread", "edges", "signs"])
@pytest.mark.parametrize("d", [2, 3, 4])
def test_f64_integer_collision_against_exact(d, kind):
    N = SHAPES[d]
    rng = np.random.default_rng(100 * d + len(kind))
    dx = 1.0 / N[0]
    eps = {2: 0.2048, 3: 0.0512, 4: 0.08}[d]
    s = lb.Solver(d, N, 0.02, dx, eps * dx * dx / 0.02)
    p = dict(s.params)
    p["sigma"] = 2.0 * p["w1"] + 4.0 * (d - 1) * p["wd"]
    q = int(p["q"])
    pitch, slab, eb = s.state_layout()
    rows = int(np.prod(N[1:]))
    w = np.array([p["w0"]] + [p["w1"]] * (2 * d) + [p["wd"]] * (q - 1 - 2 * d))
    # pre-collision populations f_i(x), q x nodes
    n = rows * N[0]
    theta = 1.0 + rng.random(n)
    f = w[:, None] * theta * (1.0 + 0.2 * rng.standard_normal((q, n)))
    if kind == "spread":  # exponents around and beyond the alignment width
        f = f * 2.0 ** -rng.integers(0, 16, size=(q, n))
    elif kind == "signs":
        f = f * rng.choice([-1.0, 1.0], size=(q, n))
    elif kind == "edges":
        f[:, 0::7] = 0.0
        f[rng.integers(0, q, n // 7), np.arange(n // 7) * 7 + 1] = 0.0
        f[:, 2::7] *= 2.0 ** -1000
        f[:, 3::7] *= 5e-324
        f[:, 4::7] = np.nextafter(2.0, 1.0)  # every magnitude at the top of its binade
        f[0, 5::14] = np.inf
        f[0, 12::14] = np.nan
        f[:, 6::7] *= 2.0 ** 1000
    e = _velocities(d)
    grid = f.reshape((q,) + tuple(reversed(N)))
    P = np.empty_like(grid)  # P_i(x - e_i) = f_i(x)
    for i in range(q):
        P[i] = np.roll(grid[i], [-v for v in e[i]], [d - 1 - a for a in range(d)])
    buf = np.zeros((q, rows, pitch))
    buf[:, :, :N[0]] = P.reshape(q, rows, N[0])
    s.load_state(torch.from_numpy(buf).cuda().view(torch.uint8), 0)
    s.step(1)
    got = s.save_state().cpu().numpy().view(np.float64).reshape(q, rows, pitch)[:, :, :N[0]].reshape(q, n)
    tight = 0
    for x in range(n):
        col = f[:, x]
        if not np.all(np.isfinite(col)):
            assert not np.all(np.isfinite(got[:, x]))
            continue
        exact = _collide_exact([Fraction(float(v)) for v in col], d, p)
        total = sum(abs(Fraction(float(v))) for v in col)
        ex = np.frexp(np.abs(col))[1]
        # normal numbers within the width and a sum well inside the limit
        sure = np.all(col != 0) and ex.max() - ex.min() <= WIDTH[d] and -900 < ex.min() and ex.max() < 900 and \
            total * 2 ** (52 + WIDTH[d]) < Fraction(2) ** (61 + int(ex.max()) - 1)
        tight += bool(sure)
        for i in range(q):
            v = got[i, x]
            if not np.isfinite(v):  # 2^1000-scaled sums stay finite; nothing else may overflow
                raise AssertionError((kind, x, i, v))
            err = abs(Fraction(float(v)) - exact[i])
            tiny = Fraction(16) * Fraction(5e-324)
            if sure:
                # one rounding of the result; up to q + 2 products, each off by at most two units of the
                # aligned values; and the host's rounding of the constants (a few 2^-54 of each)
                unit = Fraction(2) ** (int(ex.max()) - 1 - 52 - WIDTH[d])
                assert err <= abs(exact[i]) / 2 ** 53 + 2 * (q + 2) * unit + total / 2 ** 54 * 8, (kind, x, i)
            assert err <= 16 * total / 2 ** 53 + tiny, (kind, x, i)
    if kind == "run":
        assert tight > n // 2
    s.close()
