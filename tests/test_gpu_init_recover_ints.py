"""The recovery's quotient, formed on the integer pipes, against IEEE division."""

import numpy as np
import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu


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
