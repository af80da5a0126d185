"""Solvers beyond one page-locked slab (64), made, used and closed out of order
and from several threads: each reads its own results."""

import threading

import pytest
import torch

from paper_2309_02825_gb300 import lb

pytestmark = pytest.mark.gpu


def _solver(k):
    n = 16 + k % 5
    s = lb.Solver(2, (n, n), 0.02, 1.0 / n, 0.2048 / n**2 / 0.02, precision="fp64")
    th = torch.full((n, n), 1.0 + k, dtype=torch.float64, device="cuda")
    s.set_theta0(th, torch.zeros((2, n, n), dtype=torch.float64, device="cuda"))
    return s, (1.0 + k) * n * n


def test_results_of_many_live_solvers():
    live = [_solver(k) for k in range(150)]
    torch.cuda.synchronize()
    for s, want in live[::-1]:
        assert s.sum_theta() == pytest.approx(want, rel=1e-14)
    for s, _ in live[::2]:
        s.close()
    kept = live[1::2] + [_solver(200 + k) for k in range(80)]
    for s, want in kept:
        assert s.sum_theta() == pytest.approx(want, rel=1e-14)
    for s, _ in kept:
        s.close()


def test_results_from_threads():
    bad = []

    def work(t):
        for k in range(20):
            s, want = _solver(10 * t + k)
            if abs(s.sum_theta() - want) > 1e-13 * want:
                bad.append((t, k))
            s.close()

    threads = [threading.Thread(target=work, args=(t,)) for t in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
