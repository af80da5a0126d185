"""FP64 rows that leave lanes of a warp without a node: the sweep costs what it
costs on full rows of a node more."""

import time

import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu


def _us_per_sweep(N, eps):
    d = len(N)
    dx = 1.0 / N[0]
    s = lb.Solver(d, N, 0.02, dx, eps * dx * dx / 0.02, precision="fp64")
    shape = tuple(reversed(N))
    s.set_theta0(torch.full(shape, 1.5, dtype=torch.float64, device="cuda"),
                 torch.zeros((d,) + shape, dtype=torch.float64, device="cuda"))
    s.step(64)
    best = 1e30
    for _ in range(5):
        torch.cuda.synchronize()
        t = time.perf_counter()
        s.step(64)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    s.close()
    return best / 64 * 1e6


@pytest.mark.parametrize("ragged,full,eps", [((63, 120, 120), (64, 120, 120), 0.0512),
                                             ((127, 120, 120), (128, 120, 120), 0.0512),
                                             ((31, 30, 30, 30), (32, 30, 30, 30), 0.08)])
def test_lanes_beyond_the_row_cost_nothing(ragged, full, eps):
    """The same warps and nearly the same bytes; lanes that ran the direct form beside
    the others' integer form took 1.3 to 2.6 times as long."""
    assert _us_per_sweep(ragged, eps) < 1.2 * _us_per_sweep(full, eps)
