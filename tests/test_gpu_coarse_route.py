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
