"""Which kernel a flow product takes follows the permeabilities of the moment."""
import numpy as np
import pytest

import workloads as W

from gpu_common import cuda, need_gpu, solver_for

pytestmark = pytest.mark.gpu


def problem(k=None):
    prob = W.tiny_faulted(16, 14, 9, seed=3, h=(0.4, 0.3, 0.5))
    prob.kf = prob.fault = None
    N = prob.n_nodes
    prob.fixed = np.zeros((4, N), np.uint8)
    prob.fixed[3, -2:] = 1
    prob.fu, prob.fp = np.zeros((3, N)), np.zeros(N)
    if k is not None:
        prob.k = k
    return prob


@pytest.mark.parametrize("dt", [3.0, 1e10])
def test_solves_follow_elements_that_lose_or_gain_flow(dt):
    """Same smallest positive and largest k before and after: a solver that was given the new
    array later returns what a fresh one does, bit for bit."""
    need_gpu()
    prob = problem()
    rng = np.random.default_rng(4)
    full = 10.0 ** rng.uniform(-15.0, -14.0, prob.n_el)
    holes = full.copy()
    inner = rng.permutation(prob.n_el)[:20]
    holes[[e for e in inner if full[e] not in (full.min(), full.max())]] = 0.0
    b = cuda(rng.normal(size=prob.n_nodes) * 1e-12 * (prob.fixed[3] == 0))
    s = solver_for(problem(full))
    s.timestep(dt)
    for k in (full, holes, full):
        s.set_permeability(k)
        x, _ = s.pcg("A22", b, rtol=1e-8)
        f = solver_for(problem(k))
        f.timestep(dt)
        y, _ = f.pcg("A22", b, rtol=1e-8)
        assert bool((x == y).all())


@pytest.mark.parametrize("ratio", [2.0 ** 5, 2.0 ** 18, 2.0 ** 23, 2.0 ** 30, 2.0 ** 37, 2.0 ** 50])
def test_uniform_pressure_meets_its_storage_alone(ratio):
    """A uniform pressure moves no fluid: S p + dt C p is S p, whose rows are the nodes' shares of the
    volume over M, to FP64's rounding (eight elements, three sums and scalings each) however far
    dt k/mu lies above the storage."""
    need_gpu()
    prob = problem()
    prob.fixed[:] = 0
    prob.k = 10.0 ** np.random.default_rng(4).uniform(-15.0, -14.0, prob.n_el)
    s = solver_for(prob)
    # dt k/mu h^2 V / (V/M) = ratio for the smallest cell size
    s.timestep(ratio * min(prob.h) ** 2 * prob.mu_f / (prob.k.max() * prob.M))
    p = 1.7e6 / 3.0
    y = s.apply("A22", cuda(np.full(prob.n_nodes, p))).cpu().numpy().reshape(prob.n_planes, prob.ny + 1, prob.nx + 1)
    edge = lambda n: np.r_[0.5, np.ones(n - 2), 0.5]
    share = edge(prob.n_planes)[:, None, None] * edge(prob.ny + 1)[:, None] * edge(prob.nx + 1)
    ref = share * np.prod(np.asarray(prob.h)) / prob.M * p
    assert np.max(np.abs(y / ref - 1.0)) <= 16 * 2.0 ** -53
