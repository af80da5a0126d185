"""Small grids, whose steps lb_step batches into few launches by itself (short
1D grids resident in one block, square tiles in 2D), against one sweep per
launch: the same bits at the edges of the blocks' and tiles' sizes."""

import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu


def _run(N, precision, boundary, single, steps):
    d = len(N)
    eps = {1: 0.16, 2: 0.2048}[d]
    dx = 1.0 / N[0]
    s = lb.Solver(d, N, 0.02, dx, eps * dx * dx / 0.02, precision=precision, theta_ref=1.5, boundary=boundary)
    if single:
        s.set_blocking(0)
    g = torch.Generator(device="cuda").manual_seed(3)
    shape = tuple(reversed(N))
    s.set_theta0(1.0 + torch.rand(shape, dtype=torch.float64, device="cuda", generator=g),
                 torch.randn((d,) + shape, dtype=torch.float64, device="cuda", generator=g))
    for n in steps:
        s.step(n)
    assert s.nsteps == sum(steps)
    out = list(s.macros()) + [s.sum_theta()]
    s.check()
    s.close()
    return out


@pytest.mark.parametrize("boundary", [None, ["mirror"]])
@pytest.mark.parametrize("precision", ["fx64", "fp32s", "fp64"])
def test_resident_1d_equals_single_sweeps(precision, boundary):
    for n in (1, 2, 3, 4, 31, 32, 33, 81, 511, 1023, 1024, 1025, 1026, 2047, 2048, 2049, 4095, 4096, 4097):
        if boundary and n < 3:
            continue
        a = _run((n,), precision, boundary, False, [1, 6, 2])
        b = _run((n,), precision, boundary, True, [1, 6, 2])
        assert a[-1] == b[-1], n
        for x, y in zip(a[:-1], b[:-1]):
            assert torch.equal(x, y), n


@pytest.mark.parametrize("precision", ["fx64", "fp32s", "fp64"])
@pytest.mark.parametrize("N", [(1, 1), (3, 2), (8, 8), (9, 70), (64, 64), (96, 97), (101, 150), (250, 255), (400, 30),
                               (470, 300), (500, 500)])
def test_small_2d_equals_single_sweeps(N, precision):
    a = _run(N, precision, None, False, [1, 8, 21])
    b = _run(N, precision, None, True, [1, 8, 21])
    assert a[-1] == b[-1]
    for x, y in zip(a[:-1], b[:-1]):
        assert torch.equal(x, y)


def test_resident_1d_range_overflow_is_reported():
    """An unstable relaxation set is reported whatever the schedule."""
    relax = {"s1": 1.9, "s2x": 0.9, "w1": 0.49}
    got = []
    for single in (False, True):
        s = lb.Solver(1, (200,), 0.02, 0.005, 0.16 * 0.005**2 / 0.02, relax=relax, precision="fx64")
        if single:
            s.set_blocking(0)
        x = torch.ones(200, dtype=torch.float64, device="cuda")
        x[::2] = 2.0
        s.set_theta0(x, torch.zeros(1, 200, dtype=torch.float64, device="cuda"))
        s.step(3000)
        try:
            s.check()
            got.append(lb.LB_OK)
        except lb.LBError as e:
            got.append(e.status)
        s.close()
    assert got[0] == got[1]
