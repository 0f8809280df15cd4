"""The coarsest multigrid level as one cluster kernel: K_T solves on grids whose coarsest
level has fewer, as many and more node rows than the cluster has CTAs, is one element
layer thin, long in x or z, of every cell class, with and without a fault.

A wrong polynomial is not the symmetric positive preconditioner CG needs: the solve would
miss its tolerance or take as many iterations as block Jacobi, which the multigrid cuts by
a factor of three or more on these grids."""
import numpy as np
import pytest

import workloads as W

from gpu_common import cuda, need_gpu, solver_for, torch

pytestmark = pytest.mark.gpu

SHEARS = {"box": (0.0, 0.0), "dip": (1.7320508075688772, 0.0), "skew": (0.4, -0.3)}
GRIDS = [  # nx, ny, nz, cell, fault
    (8, 8, 8, "box", True), (8, 4, 16, "dip", True), (24, 30, 20, "skew", True), (20, 32, 24, "box", True),
    (28, 36, 24, "dip", True), (64, 20, 8, "box", False), (8, 20, 60, "skew", True)]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny,nz,cell,fault", GRIDS)
def test_solves_converge_as_multigrid_does(nx, ny, nz, cell, fault, precision):
    need_gpu()
    prob = W.tiny_faulted(nx, ny, nz, shear=SHEARS[cell], seed=11, h=(0.5, 0.5, 0.5))
    if not fault:
        prob.kf = prob.fault = None
        prob.fixed = np.zeros((4, prob.n_nodes), np.uint8)
        prob.fixed[0:3, : (nx + 1) * (ny + 1)] = 1
        prob.fu, prob.fp = np.zeros((3, prob.n_nodes)), np.zeros(prob.n_nodes)
    elif (nz // 2) % 2:
        pytest.skip("fault index is not even")
    rng = np.random.default_rng(3)
    u = rng.normal(size=(3, prob.n_nodes)) * 1e-6 * (prob.fixed[:3] == 0)
    its = {}
    for kind in (1, 0):
        s = solver_for(prob)
        s.set_preconditioner(kind)
        b = s.apply("KT", cuda(u))
        if precision == "fp64":
            x, rep = s.pcg("KT", b, rtol=1e-12)
            r = b - s.apply("KT", x)
            assert torch.linalg.norm(r) <= 1e-11 * torch.linalg.norm(b)
            its[kind] = rep["iterations"]
        else:
            prob.fu = 1e4 * rng.normal(size=u.shape) * (prob.fixed[:3] == 0) if kind == 1 else prob.fu
            s.loads(prob.fu, prob.fp)
            its[kind] = s.step(1.0, newton_rtol=1e-9, precision=1)["inner_k"]
            st = s.get_state()
            ref = st if kind == 1 else ref
            assert np.linalg.norm(st["u"] - ref["u"]) <= 1e-6 * np.linalg.norm(ref["u"])
    assert 3 * its[1] <= its[0], its


@pytest.mark.parametrize("bits", [12, 21, 23, 40])
def test_modulus_contrast_on_both_sides_of_the_rule(bits):
    """Soft lower half, 2^bits below the upper one: the FP64 cluster kernel serves a contrast
    up to 2^21, the launches the rest.  The residual bound is that of the solves above."""
    need_gpu()
    nx, ny, nz = 8, 20, 16
    prob = W.tiny_faulted(nx, ny, nz, seed=11, h=(0.5, 0.5, 0.5))
    prob.kf = prob.fault = None
    prob.fixed = np.zeros((4, prob.n_nodes), np.uint8)
    prob.fixed[0:3, : (nx + 1) * (ny + 1)] = 1
    prob.fu, prob.fp = np.zeros((3, prob.n_nodes)), np.zeros(prob.n_nodes)
    prob.E = np.full_like(prob.E, 2.0 ** 34)
    prob.E[: prob.E.size // 2] *= 2.0 ** -bits
    u = np.random.default_rng(3).normal(size=(3, prob.n_nodes)) * 1e-6 * (prob.fixed[:3] == 0)
    s = solver_for(prob)
    s.set_preconditioner(1)
    b = s.apply("KT", cuda(u))
    x, rep = s.pcg("KT", b, rtol=1e-12)
    assert torch.linalg.norm(b - s.apply("KT", x)) <= 1e-11 * torch.linalg.norm(b), rep
