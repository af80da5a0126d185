"""FP64 reverse step: seeds whose node values all lie near the top of one
binade with mixed signs, where the channel sums of the integer form are as
large as they get, against the oracle's adjoint."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2309_02825_gb300 import lb
from paper_2309_02825_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# Max-norm relative bound of the other parity tests.  FP64 rounding explains
# about 1e-14 of it (T steps of some 30 operations at 2^-53); a channel sum that
# leaves 63 bits moves a node's outputs by wd 2^64 units, tenths of the seed.
TOL = 1e-12


def _seed(kind, shape, rng):
    if kind == "outliers":  # one value against all its neighbours
        g = np.full(shape, 1.99)
        g[tuple(slice(1, None, 4) for _ in shape)] = -1.99
        return g
    if kind == "signs":  # every value at the top of a binade
        return 1.99 * 2.0**-15 * rng.choice([-1.0, 1.0], size=shape)
    return rng.standard_normal(shape)  # noise


@pytest.mark.parametrize("want_nu", [True, False])
@pytest.mark.parametrize("kind", ["outliers", "signs", "noise"])
@pytest.mark.parametrize("d,N", [(2, (41, 30)), (3, (21, 18, 14)), (3, (40, 40, 40))])
def test_fp64_reverse_step_on_seeds_of_mixed_signs(d, N, kind, want_nu):
    T = 3
    rng = np.random.default_rng(11)
    nu, eps = 0.02, {2: 0.2048, 3: 0.0512}[d]
    dx = 1.0 / N[0]
    dt = eps * dx * dx / nu
    prob = W.FourierProblem.random(d, nu, 6, 3, 0.05, 1.5, 4)
    th0 = prob.theta(N, dx)
    g = _seed(kind, tuple(reversed(N)), rng)
    m = O.Model(d, N, nu, dx, dt)
    th, _, u = m.recover(m.run(m.initialize(th0), T))
    # the oracle's loss is 1/2 |u - ut|^2 + 1/2 |theta - tt|^2: its seeds are 0 and theta - tt,
    # the latter formed again from tt here so that both sides start from the same values
    tt = th - g
    _, go, dnuo = m.adjoint(th0, u, T, theta_target=tt)
    s = lb.Solver(d, N, nu, dx, dt)
    a = lb.Adjoint(s, T, want_nu=want_nu)
    a.forward(torch.from_numpy(th0).cuda())
    a.seed(None, torch.from_numpy(np.ascontiguousarray(th - tt)).cuda())
    a.step(T)
    g0, dnu = a.result()
    a.close()
    s.close()
    # theta(T) of the two sides differs by rounding, so the oracle's own seed by up to 1e-14 of theta
    slack = 1e-14 * np.max(np.abs(th)) * max(1.0, np.max(np.abs(go)) / np.max(np.abs(g)))
    assert np.max(np.abs(g0.cpu().numpy() - go)) <= TOL * np.max(np.abs(go)) + slack
    if want_nu:
        # dL/dnu sums, over nodes and steps, lambda . (dK/deps) f times deps/dnu
        terms = T * np.sum(np.abs(g)) * np.max(np.abs(th)) * eps / nu
        assert abs(dnu - dnuo) <= TOL * terms + slack * g.size * T * np.max(np.abs(th)) * eps / nu
