"""The forward pass of the adjoint on grids that run one sweep per launch: its
checkpointed segments cost about what the same steps cost in one call."""

import time

import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu


def _best(call, reps=5):
    best = 1e30
    for _ in range(reps):
        torch.cuda.synchronize()
        t = time.perf_counter()
        call()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("N,boundary,precision", [((20000,), None, "fp32s"), ((20000,), None, "fx64"),
                                                  ((160, 128), ["mirror", "periodic"], "fp32s")])
def test_segments_are_not_launched_sweep_by_sweep(N, boundary, precision):
    """900 steps in segments of 30 (30 checkpoint copies beside) against lb_step(900),
    which replays graphs: 2.3 us a sweep, 4.1 where each is launched by itself.
    The bound lies between 1.2 and 1.8 of it."""
    d, T = len(N), 900
    dx = 1.0 / N[0]
    s = lb.Solver(d, N, 0.02, dx, 0.16 * dx * dx / 0.02, precision=precision,
                  theta_ref=1.5 if precision == "fp32s" else 0.0, boundary=boundary)
    shape = tuple(reversed(N))
    th = torch.full(shape, 1.5, dtype=torch.float64, device="cuda")
    gr = torch.zeros((d,) + shape, dtype=torch.float64, device="cuda")
    a = lb.Adjoint(s, T, checkpoint=30, want_nu=True)
    a.forward(th)
    forward = _best(lambda: a.forward(th))

    def plain():
        s.set_theta0(th, gr)
        s.step(T)
        s.macros()

    plain()
    steps = _best(plain)
    a.close()
    s.close()
    assert forward < 1.5 * steps
