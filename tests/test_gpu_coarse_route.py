"""The coarsest multigrid level on the levels its cluster kernel does not take, and against the
launches that it replaces."""
import numpy as np
import pytest

import workloads as W

from gpu_common import cuda, need_gpu, solver_for, torch

pytestmark = pytest.mark.gpu


def block(nx, ny, nz, fault=True, h=(0.5, 0.5, 0.5), shear=(0.0, 0.0)):
    prob = W.tiny_faulted(nx, ny, nz, shear=shear, seed=11, h=h)
    if not fault:
        prob.kf = prob.fault = None
        prob.fixed = np.zeros((4, prob.n_nodes), np.uint8)
        prob.fixed[0:3, : (nx + 1) * (ny + 1)] = 1
        prob.fu, prob.fp = np.zeros((3, prob.n_nodes)), np.zeros(prob.n_nodes)
    return prob


@pytest.mark.parametrize("nx,ny,nz,fault", [(4, 8, 8, True), (4, 16, 4, False), (4, 8, 16, False), (8, 4, 8, True)])
def test_solves_where_the_coarsest_level_is_one_cell_thin(monkeypatch, nx, ny, nz, fault):
    """Coarsest levels of one cell in x, in x and z, in x and y: fewer iterations than block
    Jacobi, and the residual that the solve's tolerance asks for."""
    need_gpu()
    monkeypatch.setenv("GM_MG_MIN_CELLS", "1")
    prob = block(nx, ny, nz, fault)
    u = np.random.default_rng(3).normal(size=(3, prob.n_nodes)) * 1e-6 * (prob.fixed[:3] == 0)
    its = {}
    for kind in (1, 0):
        s = solver_for(prob)
        s.set_preconditioner(kind)
        b = s.apply("KT", cuda(u))
        x, rep = s.pcg("KT", b, rtol=1e-12)
        assert torch.linalg.norm(b - s.apply("KT", x)) <= 1e-11 * torch.linalg.norm(b)
        its[kind] = rep["iterations"]
    assert its[1] < its[0], its


def one_cycle(monkeypatch, cluster, prob, b):
    """x = alpha V(b) of the first PCG iteration, and the launches that it took."""
    import paper_2410_17133_gb300 as gm
    monkeypatch.setenv("GM_MG_COARSE_CLUSTER", "1" if cluster else "0")
    s = solver_for(prob)
    s.set_preconditioner(1)
    x = torch.zeros_like(b)
    with pytest.raises(gm.GMError):
        s.pcg("KT", b, x=x, rtol=1e-14, maxit=1)            # stops at its limit, with x of one iteration
    n = s.counters()[0]
    return x.cpu().numpy(), n


SKEW, DIP = (0.4, -0.3), (1.7320508075688772, 0.0)


@pytest.mark.parametrize("nx,ny,nz,shear,fault", [
    (8, 4, 16, DIP, True), (24, 32, 20, SKEW, True), (20, 36, 24, (0.0, 0.0), True), (8, 20, 60, SKEW, False)])
def test_one_launch_equals_the_launches(monkeypatch, nx, ny, nz, shear, fault):
    """The degree-24 polynomial in one launch against its 47 launches, FP64.  Each of the 24 steps
    adds about 60 roundings of its terms, which the polynomial (interval ends 383 apart) amplifies
    at most 20-fold: 24 * 60 * 20 eps < 1e-11."""
    need_gpu()
    prob = block(nx, ny, nz, fault, shear=shear)
    b = cuda(np.random.default_rng(5).normal(size=(3, prob.n_nodes)) * (prob.fixed[:3] == 0))
    (x, n), (y, m) = (one_cycle(monkeypatch, c, prob, b) for c in (True, False))
    assert m - n >= 46, (n, m)                              # one launch was taken
    assert np.linalg.norm(x - y) <= 1e-11 * np.linalg.norm(y)


@pytest.mark.parametrize("bits,cluster", [(12, True), (20, True), (23, False), (40, False)])
def test_contrast_beyond_the_rule_keeps_the_launches(monkeypatch, bits, cluster):
    need_gpu()
    prob = block(8, 20, 16, False)
    prob.E = np.full_like(prob.E, 2.0 ** 34)
    prob.E[: prob.E.size // 2] *= 2.0 ** -bits
    b = cuda(np.random.default_rng(5).normal(size=(3, prob.n_nodes)) * (prob.fixed[:3] == 0))
    (x, n), (y, m) = (one_cycle(monkeypatch, c, prob, b) for c in (True, False))
    assert (m - n >= 46) == cluster and (cluster or np.array_equal(x, y))


def test_iterations_in_single_precision_do_not_depend_on_the_route(monkeypatch):
    """FP32-refined steps both ways: the same Newton iterations, inner iterations within a tenth,
    fields within the step's tolerance."""
    need_gpu()
    out = []
    for cluster in ("1", "0"):
        monkeypatch.setenv("GM_MG_COARSE_CLUSTER", cluster)
        s = solver_for(block(20, 32, 24, True))
        rep = s.step(1.0, newton_rtol=1e-9, precision=1)
        out.append((rep["newton"], rep["inner_k"], s.counters()[0], s.get_state()["u"]))
    (n0, k0, l0, u0), (n1, k1, l1, u1) = out
    assert n0 == n1 and abs(k0 - k1) <= 0.1 * k1 and l0 < l1
    assert np.linalg.norm(u0 - u1) <= 1e-6 * np.linalg.norm(u1)


@pytest.mark.parametrize("shear", [(0.0, 0.0), DIP, SKEW])
def test_values_far_below_the_largest_keep_their_bits(monkeypatch, shear):
    """Two patches of forces, one 2^-40 of the other, on rows that one CTA owns, and polynomials so
    short that neither reaches the other: around the small patch both routes agree within some
    ten roundings of 24 products each, 500 eps < 1e-13 of the values there."""
    need_gpu()
    monkeypatch.setenv("GM_MG_COARSE_DEG", "2")
    monkeypatch.setenv("GM_MG_SMOOTH_DEG", "1")
    prob = block(8, 20, 60, False, shear=shear)
    k = np.arange(prob.n_nodes) // (9 * 21)
    size = np.where(abs(k - 10) <= 1, 1.0, 0.0) + np.where(abs(k - 50) <= 1, 2.0 ** -40, 0.0)
    b = cuda(np.random.default_rng(5).normal(size=(3, prob.n_nodes)) * size)
    (x, n), (y, m) = (one_cycle(monkeypatch, c, prob, b) for c in (True, False))
    assert m - n >= 2                                       # degree 2: three launches in one
    far = k >= 40
    assert np.abs(y[:, far]).max() > 0.0
    assert np.abs(x - y)[:, far].max() <= 1e-13 * np.abs(y[:, far]).max()
