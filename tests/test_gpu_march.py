"""Sweeps of several steps per launch that lb_step takes by itself on large
periodic grids (marching windows) against one sweep per launch: the same bits,
over window and chunk remainders, steps that do not fill a launch, and both
recoveries' inputs (the state and the conserved total)."""

import numpy as np
import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu

# one window exactly, one column more, one less; ragged; a last chunk of few rows; long rows
GRIDS_2D = [(60, 4000), (61, 4001), (59, 4003), (120, 2100), (501, 443), (2113, 201), (124, 1999), (125, 2000),
            (1500, 1301)]
GRIDS_3D = [(30, 11, 1000), (31, 12, 1001), (29, 23, 500), (28, 12, 3601), (29, 13, 3200), (57, 25, 900), (101, 90, 140)]


def _pair(d, N, precision, relax=None):
    eps = {2: 0.2048, 3: 0.0512}[d]
    dx = 1.0 / N[0]
    nu = 0.02
    out = []
    for single in (False, True):
        s = lb.Solver(d, N, nu, dx, eps * dx * dx / nu, relax=relax, precision=precision, theta_ref=1.5)
        if single and d == 2:
            s.set_blocking(0)
        out.append(s)
    return out


def _inputs(d, N):
    g = torch.Generator(device="cuda").manual_seed(7)
    shape = tuple(reversed(N))
    th = 1.0 + torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)
    gr = torch.randn((d,) + shape, dtype=torch.float64, device="cuda", generator=g)
    return th, gr


@pytest.mark.parametrize("precision", ["fx64", "fp32s", "fp64"])
@pytest.mark.parametrize("N", GRIDS_2D + GRIDS_3D)
def test_marching_equals_single_sweeps(N, precision):
    d = len(N)
    auto, single = _pair(d, N, precision)
    th, gr = _inputs(d, N)
    steps = [1, 13, 2]
    for s in (auto, single):
        s.set_theta0(th, gr)
    for n in steps:
        auto.step(n)
        if d == 2:
            single.step(n)
        else:
            for _ in range(n):  # one step per call: one sweep per launch
                single.step(1)
        assert auto.nsteps == single.nsteps
    assert auto.sum_theta() == single.sum_theta()
    for a, b in zip(auto.macros(), single.macros()):
        assert torch.equal(a, b)
    for s in (auto, single):
        s.check()
        s.close()


def test_marching_fx64_range_overflow_is_reported():
    """Every step's values are checked: an unstable relaxation set is reported
    (LB_EINVAL) on a grid that marches, as with one sweep per launch."""
    N = (512, 431)
    relax = {"s1": 1.46, "s2x": 1.07, "s22": 0.69, "w1": 0.29, "wd": -0.01}  # grows by 1.34 per step
    auto, single = _pair(2, N, "fx64", relax)
    th, gr = _inputs(2, N)
    states = []
    for s in (auto, single):
        s.set_theta0(th, 0 * gr)
        s.step(402)
        with pytest.raises(lb.LBError) as ei:
            s.check()
        states.append(ei.value.status)
        s.close()
    assert states == [lb.LB_EINVAL, lb.LB_EINVAL]


def test_marching_inside_a_captured_graph():
    N = (700, 613)
    auto, single = _pair(2, N, "fx64")
    th, gr = _inputs(2, N)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()  # the inputs were made on another stream
    dx = 1.0 / N[0]
    s = lb.Solver(2, N, 0.02, dx, 0.2048 * dx * dx / 0.02, precision="fx64", stream=stream)
    with torch.cuda.stream(stream):
        s.set_theta0(th, gr)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            s.step(14)
        g.replay()
        got = s.macros()
    single.set_theta0(th, gr)
    single.step(14)
    torch.cuda.synchronize()
    for a, b in zip(got, single.macros()):
        assert torch.equal(a, b)
    for x in (s, auto, single):
        x.close()


@pytest.mark.parametrize("d,N,prec", [(1, (81,), "fx64"), (2, (64, 50), "fx64"), (2, (700, 613), "fx64"),
                                      (2, (1201, 1000), "fp32s"), (3, (101, 90, 77), "fp32s")])
@pytest.mark.parametrize("n", [1, 8, 14, 17])
def test_captured_steps_replay_one_after_another(d, N, prec, n):
    """An even captured call, or an odd one captured twice, ends in the buffer it
    began in, whatever the number of steps of a launch: replays continue."""
    th, gr = _inputs(d, N)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    dx = 1.0 / N[0]
    eps = 0.0512 if d == 3 else 0.2048
    s = lb.Solver(d, N, 0.02, dx, eps * dx * dx / 0.02, precision=prec, theta_ref=1.5, stream=stream)
    calls = 1 + n % 2
    with torch.cuda.stream(stream):
        s.set_theta0(th, gr)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            for _ in range(calls):
                s.step(n)
        for _ in range(3):
            g.replay()
        got = s.macros()
        s.set_theta0(th, gr)
        for _ in range(3 * calls * n):
            s.step(1)
        want = s.macros()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    s.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32s", "fx64"])
def test_captured_batch_steps_replay_one_after_another(prec):
    sizes = [(130, 96), (257, 201)]
    dx = [1.0 / n[0] for n in sizes]
    stream = torch.cuda.Stream()
    ins = [_inputs(2, n) for n in sizes]
    th = torch.cat([t.reshape(-1) for t, _ in ins])
    gr = torch.cat([g.reshape(-1) for _, g in ins])
    torch.cuda.synchronize()
    kw = {"theta_ref": [1.5, 1.5]} if prec == "fp32s" else {}
    b = lb.Batch(sizes, [0.02] * 2, dx, [0.2048 * x * x / 0.02 for x in dx], precision=prec, stream=stream, **kw)
    with torch.cuda.stream(stream):
        b.set_theta0(th, gr)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            b.step(14)
        for _ in range(3):
            g.replay()
        got = b.macros()
        b.set_schedule(1e18, 128, False)
        b.set_theta0(th, gr)
        b.step(42)
        want = b.macros()
    torch.cuda.synchronize()
    for x, y in zip(got, want):
        assert torch.equal(x, y)
    b.close()


def test_blocking_call_still_selects_single_sweeps():
    s = lb.Solver(2, (600, 500), 0.02, 1.0 / 600, 0.2048 / 600**2 / 0.02, precision="fx64")
    assert s.blocking()["steps_per_launch"] == 0
    s.set_blocking(4, 24, 256)
    assert s.blocking()["steps_per_launch"] == 4
    s.set_blocking(0)
    assert s.blocking()["steps_per_launch"] == 0
    s.close()
