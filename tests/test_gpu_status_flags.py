"""Status flags of calls whose field has gone bad everywhere: reported by the
call that meets them, each time and only then, and at the cost of a good call."""

import time

import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu


def _solver(n, precision):
    s = lb.Solver(2, (n, n), 0.02, 1.0 / n, 0.2048 / n**2 / 0.02, precision=precision,
                  theta_ref=1.5 if precision == "fp32s" else 0.0)
    th = torch.full((n, n), 1.5, dtype=torch.float64, device="cuda")
    th[::2] = 1.25
    return s, th, torch.zeros((2, n, n), dtype=torch.float64, device="cuda")


def _bad_state(s, precision):
    buf = s.save_state()
    if precision == "fp32s":
        buf.view(torch.float32).fill_(-1.0)  # theta = theta_ref - 9
    else:
        buf.zero_()  # theta = 0
    return buf


def _status(call):
    try:
        call()
    except lb.LBError as e:
        return e.status
    return lb.LB_OK


@pytest.mark.parametrize("precision", ["fp64", "fp32s", "fx64"])
def test_bad_fields_are_reported_each_time_and_only_then(precision):
    s, th, gr = _solver(70, precision)
    for _ in range(2):
        assert _status(lambda: s.set_theta0(-th, gr)) == lb.LB_ENONPOS
        assert _status(lambda: s.set_theta0(th, gr)) == lb.LB_OK
        good, bad = s.save_state(), _bad_state(s, precision)
        s.load_state(bad, 3)
        first = _status(s.macros)
        assert first != lb.LB_OK
        s.load_state(good, 0)
        assert _status(s.macros) == lb.LB_OK
        s.load_state(bad, 3)
        assert _status(s.macros) == first
        s.load_state(bad, 3)
        s.load_state(good, 0)
        s.step(2)
        assert _status(s.macros) == lb.LB_OK
        assert _status(s.check) == lb.LB_OK
    s.close()


def _best_us(call, reps=5):
    best = 1e30
    for _ in range(reps):
        torch.cuda.synchronize()
        t = time.perf_counter()
        call()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t)
    return best * 1e6


@pytest.mark.parametrize("precision", ["fp64", "fp32s", "fx64"])
def test_a_bad_field_costs_no_more_than_a_good_one(precision):
    """The warps' flags stay on the device but for the first (each one over the
    host link took 10 to 20 times a good call's time at this size)."""
    s, th, gr = _solver(2048, precision)
    neg = -th
    good = _best_us(lambda: s.set_theta0(th, gr))
    bad = _best_us(lambda: _status(lambda: s.set_theta0(neg, gr)))
    s.close()
    assert bad < 3.0 * good
