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


def _rough(N, seed=7):
    """Random theta in [1, 2) and a random gradient: FP64 nodes of both forms."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = tuple(reversed(N))
    return (1.0 + torch.rand(shape, dtype=torch.float64, device="cuda", generator=g),
            torch.randn((len(N),) + shape, dtype=torch.float64, device="cuda", generator=g))


# windows of 60, 120 and 126 columns (fixed point, FP32, FP64), 30 and 28 in 3D: whole
# windows, one column more (a column fewer each and a narrow last one) and one less; last
# chunks of any number of rows
@pytest.mark.parametrize("precision,N", [
    ("fx64", (60, 8000)), ("fx64", (600, 800)), ("fx64", (601, 801)), ("fx64", (599, 803)), ("fx64", (1501, 443)),
    ("fp32s", (120, 4000)), ("fp32s", (1200, 400)), ("fp32s", (1201, 401)), ("fp32s", (1199, 403)),
    ("fp32s", (2113, 301)), ("fp64", (126, 15000)), ("fp64", (1512, 1300)), ("fp64", (1511, 1303)),
    ("fp64", (251, 7503)), ("fx64", (60, 44, 200)), ("fx64", (61, 45, 201)), ("fx64", (59, 43, 203)),
    ("fx64", (30, 33, 500)), ("fx64", (29, 23, 700)), ("fp32s", (56, 48, 300)), ("fp32s", (57, 49, 301)),
    ("fp32s", (55, 47, 299)), ("fp32s", (85, 61, 201)), ("fp32s", (57, 25, 900))])
def test_marching_windows_give_the_bits_of_single_sweeps(precision, N, tmp_path):
    th, gr = _rough(N)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = _solver(N, precision, stream=stream)
    one = _solver(N, precision)
    if len(N) == 2:
        one.set_blocking(0)
    s.set_theta0(th, gr)
    assert "march" in _steps(s, stream, 13, tmp_path)
    s.set_theta0(th, gr)
    one.set_theta0(th, gr)
    for n in (13, 1, 6):
        s.step(n)
        for _ in range(n):  # one step per call: one sweep per launch
            one.step(1)
    torch.cuda.synchronize()
    assert s.sum_theta() == one.sum_theta()
    got = s.macros()
    torch.cuda.synchronize()
    for a, b in zip(got, one.macros()):
        assert torch.equal(a, b)
    s.check()
    s.close()
    one.close()


@pytest.mark.parametrize("precision", ["fx64", "fp32s", "fp64"])
def test_marching_batches_give_the_bits_of_one_launch_per_step(precision, tmp_path):
    """Instances smaller than a window, of one to three rows, and a column more or
    less than one, two and three windows (60, 56 and 126 columns), beside ones
    large enough for the batch to march."""
    edge = {"fx64": 60, "fp32s": 56, "fp64": 126}[precision]
    sizes = [(1, 1), (2, 3), (5, 1), (7, 2), (edge, 3), (edge - 1, 40), (edge + 1, 41), (2 * edge, 9), (2 * edge + 1, 17),
             (2 * edge - 1, 16), (3 * edge + 1, 8), (33, 500), (1500, 1100)]
    ins = [_rough(N, 3 + k) for k, N in enumerate(sizes)]
    th = torch.cat([t.reshape(-1) for t, _ in ins])
    gr = torch.cat([g.reshape(-1) for _, g in ins])
    dx = [1.0 / N[0] for N in sizes]
    kw = {"theta_ref": [1.5] * len(sizes)} if precision == "fp32s" else {}
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    out = []
    for own in (True, False):
        b = lb.Batch(sizes, [NU] * len(sizes), dx, [EPS[2] * h * h / NU for h in dx], precision=precision, stream=stream,
                     **kw)
        if not own:
            b.set_schedule(1e18, 128)
        b.set_theta0(th, gr)
        assert ("march_batch" in _steps(b, stream, 13, tmp_path)) == own
        b.set_theta0(th, gr)
        for n in (13, 1, 6):
            b.step(n)
        out.append(b.macros())
        torch.cuda.synchronize()
        b.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("single", [False, True])
def test_resident_1d_reports_an_unstable_relaxation_set(single, tmp_path):
    """w1 = 0.7 with s2 = 0.6 grows by 1.37 a step (largest eigenvalue over the wave
    numbers): reported whatever the schedule."""
    stream = torch.cuda.Stream()
    s = lb.Solver(1, (200,), NU, 0.005, 0.16 * 0.005**2 / NU, relax={"s1": 1.5, "s2x": 0.6, "w1": 0.7}, precision="fx64",
                  stream=stream)
    if single:
        s.set_blocking(0)
    x = torch.ones(200, dtype=torch.float64, device="cuda")
    x[::2] = 2.0
    torch.cuda.synchronize()
    s.set_theta0(x, torch.zeros(1, 200, dtype=torch.float64, device="cuda"))
    assert _steps(s, stream, 5, tmp_path) == (["sweep"] * 5 if single else ["line"])
    # (the captured call did not run, and an odd number of launches ends in the other buffer)
    s.set_theta0(x, torch.zeros(1, 200, dtype=torch.float64, device="cuda"))
    s.step(400)
    with pytest.raises(lb.LBError) as ei:
        s.check()
    assert ei.value.status == lb.LB_EINVAL
    s.close()


@pytest.mark.parametrize("precision,N", [("fx64", (263, 1052)), ("fp32s", (101, 90, 77)), ("fp32s", (79, 79, 79)),
                                         ("fx64", (169, 169, 11))])
def test_graphs_of_sweeps_with_marching_remainders_give_the_same_bits(precision, N, tmp_path):
    """Grids whose windows pay only against sweeps launched one by one: calls of a
    graph's 32 steps and more replay sweeps and march the rest; captured calls sweep."""
    th, gr = _rough(N)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = _solver(N, precision, stream=stream)
    one = _solver(N, precision)
    s.set_theta0(th, gr)
    assert set(_steps(s, stream, 30, tmp_path)) == {"sweep"}
    s.set_theta0(th, gr)
    one.set_theta0(th, gr)
    for n in (13, 45, 2, 64, 31):
        s.step(n)
        for _ in range(n):
            one.step(1)
    assert s.nsteps == one.nsteps
    torch.cuda.synchronize()
    assert s.sum_theta() == one.sum_theta()
    got = s.macros()
    torch.cuda.synchronize()
    for a, b in zip(got, one.macros()):
        assert torch.equal(a, b)
    s.check()
    s.close()
    one.close()


@pytest.mark.parametrize("precision,count,edge", [("fp32s", 11, 68), ("fx64", 43, 69), ("fp64", 90, 64)])
def test_batches_mix_graphs_and_marching_remainders_bit_for_bit(precision, count, edge):
    """Batches near where marching pays: calls shorter and longer than a recorded graph of
    one launch per step, against one launch per step throughout."""
    sizes = [(edge + 3 * (j % 5) - 6, edge + 2 * (j % 7) - 6) for j in range(count)]
    ins = [_rough(N, 3 + k) for k, N in enumerate(sizes)]
    th = torch.cat([t.reshape(-1) for t, _ in ins])
    gr = torch.cat([g.reshape(-1) for _, g in ins])
    dx = [1.0 / N[0] for N in sizes]
    kw = {"theta_ref": [1.5] * count} if precision == "fp32s" else {}
    out = []
    for own in (True, False):
        b = lb.Batch(sizes, [NU] * count, dx, [EPS[2] * h * h / NU for h in dx], precision=precision, **kw)
        if not own:
            b.set_schedule(1e18, 128)
        b.set_theta0(th, gr)
        for n in (13, 45, 2, 64, 31):
            b.step(n)
        out.append(b.macros())
        b.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
