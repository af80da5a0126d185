"""Which launches lb_step and lb_batch_step take by themselves: read from the
kernels of a captured call, and the same bits as one sweep per launch."""

import re

import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]

EPS = {1: 0.16, 2: 0.2048, 3: 0.0512}
NU = 0.02


def _solver(N, precision, eps=None, stream=None, boundary=None):
    d = len(N)
    dx = 1.0 / N[0]
    return lb.Solver(d, N, NU, dx, (eps or EPS[d]) * dx * dx / NU, precision=precision,
                     theta_ref=1.5 if precision == "fp32s" else 0.0, stream=stream, boundary=boundary)


def _inputs(N, seed=3):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = tuple(reversed(N))
    th = 1.0 + torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)
    return th, torch.zeros((len(N),) + shape, dtype=torch.float64, device="cuda")


def _kernels(stream, call, tmp_path):
    """Names of the kernels that a call launches, from its captured graph."""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    with torch.cuda.graph(g, stream=stream):
        call()
    path = str(tmp_path / "graph.dot")
    g.debug_dump(path)
    with open(path) as f:
        return re.findall(r"_ZN3lbk\d+(\w+?)_kernelI", f.read())


def _steps(s, stream, n, tmp_path):
    torch.cuda.synchronize()  # the inputs were made on another stream
    with torch.cuda.stream(stream):
        names = _kernels(stream, lambda: s.step(n), tmp_path)
    torch.cuda.synchronize()
    return names


@pytest.mark.parametrize("N,several", [((96, 96), "batch_tb"), ((256, 256), "batch_tb"), ((1408, 1408), "march")])
def test_fp64_takes_several_steps_per_launch_where_its_collisions_align(N, several, tmp_path):
    """Populations near w_i theta align at eps = 0.2048, not at 0.01 (weights a
    factor 200 apart) nor at 1/2 (a weight vanishes): there one sweep per launch,
    but for the smallest grids, also after a change of the viscosity."""
    stream = torch.cuda.Stream()
    th, gr = _inputs(N)
    s = _solver(N, "fp64", stream=stream)
    one = _solver(N, "fp64", stream=stream)
    one.set_blocking(0)
    for eps in (0.2048, 0.01, 0.5, 0.2048):
        for x in (s, one):
            x.set_viscosity(NU * eps / 0.2048)
            x.set_theta0(th, gr)
        direct = "batch_tb" if N == (96, 96) else "sweep"
        names = set(_steps(s, stream, 7, tmp_path))
        assert several in names if eps == 0.2048 else names == {direct}
        assert set(_steps(one, stream, 7, tmp_path)) == {"sweep"}
        for x in (s, one):
            x.set_theta0(th, gr)
            x.step(21)
        for a, b in zip(s.macros(), one.macros()):
            assert torch.equal(a, b)
    s.close()
    one.close()


@pytest.mark.parametrize("N,precision,n,want", [
    ((81,), "fp64", 1, "sweep"), ((81,), "fp64", 3, "line"), ((2048,), "fp64", 1, "sweep"), ((2048,), "fp64", 3, "line"),
    ((4096,), "fp32s", 1, "sweep"), ((4096,), "fp32s", 3, "line"), ((4096,), "fx64", 1, "sweep"),
    ((4096,), "fx64", 4, "sweep"), ((4096,), "fx64", 5, "line"), ((256, 256), "fp32s", 1, "sweep"),
    ((256, 256), "fp32s", 3, "batch_tb"), ((416, 416), "fp32s", 1, "sweep"), ((416, 416), "fp32s", 2, "sweep"),
    ((416, 416), "fp32s", 3, "batch_tb"), ((416, 416), "fx64", 1, "sweep"), ((416, 416), "fx64", 7, "batch_tb")])
def test_calls_of_few_steps_take_single_sweeps(N, precision, n, want, tmp_path):
    """A launch of several steps costs more than the sweeps of a short call."""
    stream = torch.cuda.Stream()
    s = _solver(N, precision, stream=stream)
    s.set_theta0(*_inputs(N))
    assert set(_steps(s, stream, n, tmp_path)) == {want}
    s.close()


@pytest.mark.parametrize("N,precision", [((4096,), "fx64"), ((2048,), "fp64"), ((416, 416), "fp32s"), ((96, 97), "fx64")])
@pytest.mark.parametrize("n", [2, 6, 9, 10, 14, 18])
def test_replays_of_mixed_launches_go_on_from_one_another(N, precision, n):
    """Even captured calls (odd ones twice) end in the buffer they began in where a
    call mixes launches of several steps and single sweeps."""
    th, gr = _inputs(N)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = _solver(N, precision, stream=stream)
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


@pytest.mark.parametrize("count,N,precision,eps,march", [
    (976, (512, 2), "fp32s", None, False), (122, (512, 16), "fp32s", None, True), (1953, (512, 1), "fx64", None, False),
    (31, (2000, 16), "fx64", None, True), (200, (64, 64), "fp64", None, False), (4, (1024, 1024), "fp64", None, True),
    (4, (1024, 1024), "fp64", 0.01, False)])
def test_batches_march_where_the_windows_pay(count, N, precision, eps, march, tmp_path):
    dx = 1.0 / N[0]
    stream = torch.cuda.Stream()
    kw = {"theta_ref": [1.5] * count} if precision == "fp32s" else {}
    b = lb.Batch([N] * count, [NU] * count, [dx] * count, [(eps or EPS[2]) * dx * dx / NU] * count, precision=precision,
                 stream=stream, **kw)
    nodes = count * N[0] * N[1]
    b.set_theta0(torch.full((nodes,), 1.25, dtype=torch.float64, device="cuda"),
                 torch.zeros(2 * nodes, dtype=torch.float64, device="cuda"))
    assert ("march_batch" in _steps(b, stream, 10, tmp_path)) == march
    b.close()


@pytest.mark.parametrize("N,precision,want", [
    ((512, 512), "fx64", "march"), ((526, 526), "fx64", "march"), ((263, 1052), "fx64", "sweep"),
    ((448, 448), "fx64", "batch_tb"), ((526, 526), "fp32s", "march"), ((6036, 30), "fp32s", "batch_tb"),
    ((427, 427), "fp32s", "batch_tb"), ((126, 31, 126), "fp32s", "sweep"), ((234, 234, 15), "fp32s", "sweep"),
    ((50, 200, 50), "fp32s", "march"), ((106, 106, 106), "fp32s", "march"), ((169, 169, 11), "fx64", "sweep"),
    ((72, 72, 72), "fx64", "march"), ((1408, 1408), "fp64", "march")])
def test_grids_march_where_the_windows_pay(N, precision, want, tmp_path):
    stream = torch.cuda.Stream()
    s = _solver(N, precision, stream=stream)
    s.set_theta0(*_inputs(N))
    names = set(_steps(s, stream, 30, tmp_path))
    assert want in names and (want != "sweep" or names == {"sweep"})
    s.close()
