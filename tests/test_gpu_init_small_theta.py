"""FP32 initialisation where theta is very near its reference beside a steep
gradient: the populations that the gradient does not enter keep the accuracy of
their own terms."""

import numpy as np
import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu

SHAPES = {1: (301,), 2: (67, 41), 3: (13, 11, 9), 4: (7, 6, 5, 5)}
EPS = {1: 0.16, 2: 0.2048, 3: 0.0512, 4: 0.08}


@pytest.mark.parametrize("d", [1, 2, 3, 4])
@pytest.mark.parametrize("away", [2.0**-45, 2.0**-20, 0.0])
def test_populations_without_the_gradient_are_rounded_once(d, away):
    """f_0 = w0 (theta - theta_ref), and w1 (theta - theta_ref) along the axes that
    the gradient does not point along: one rounding to FP32 (2^-24) after
    products in 53 bits or more."""
    N = SHAPES[d]
    shape = tuple(reversed(N))
    rng = np.random.default_rng(d)
    th = 1.5 + away * rng.integers(-9, 10, shape)
    g = np.zeros((d,) + shape)
    g[0] = 1e5 * rng.standard_normal(shape)
    dx = 1.0 / N[0]
    s = lb.Solver(d, N, 0.02, dx, EPS[d] * dx * dx / 0.02, precision="fp32s", theta_ref=1.5)
    s.set_theta0(torch.from_numpy(th).cuda(), torch.from_numpy(g).cuda())
    pitch, slab, _ = s.state_layout()
    p = s.params
    buf = s.save_state().cpu().numpy().view(np.float32)
    s.close()
    rows = int(np.prod(N[1:]))
    dth = (th - 1.5).astype(np.longdouble)
    for i in [0] + [1 + a for a in range(1, d)] + [1 + d + a for a in range(1, d)]:
        got = buf[i * slab:i * slab + rows * pitch].reshape(rows, pitch)[:, :N[0]].reshape(shape).astype(np.longdouble)
        f = np.longdouble(p["w1"] if i else p["w0"]) * dth
        if i:  # stored at x - e_i
            f = np.roll(f, -1 if i <= d else 1, d - 1 - (i - 1) % d)
        assert np.all(np.abs(got - f) <= np.abs(f) * np.longdouble(2.0)**-24 * (1 + 2.0**-20)), i
