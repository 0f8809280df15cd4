"""The K solves of a tetrahedral step as one launch of one block per SM: meshes of one
block, of two, with an odd number of rows in the last block, with several passes over a
block's rows, and one whose rows no longer fit (the solve of two launches per iteration).

The step's equations are checked with the oracle's matrices.  K is solved to 1e-12 of its
right-hand side and the pressure system to 1e-10 of its first residual; rounding in the
recursions adds about eps times the condition number (1e4 at most here), so 1e-9 of the
force terms and 1e-8 of the volume terms."""
import numpy as np
import pytest

import workloads as W
from oracle import tet

from gpu_common import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 7, 13, 24, 28])
def test_steps_satisfy_their_equations(n):
    need_gpu()
    import paper_2410_17133_gb300 as gm
    prob = W.cryer_octant(n=n, steps=10)
    m = tet.TetModel(prob)
    s = gm.TetSolver.from_problem(prob)
    u = torch.zeros((3, m.N), dtype=torch.float64, device="cuda")
    p = torch.zeros(m.N, dtype=torch.float64, device="cuda")
    u0, p0 = np.zeros(3 * m.N), np.zeros(m.N)
    for dt in prob.dts[4:6]:
        s.step(dt, u, p, rtol=1e-10)
        u1, p1 = u.cpu().numpy().reshape(-1), p.cpu().numpy()
        terms = [m.Kb @ u1, m.Apu @ p1, m.fu]
        r = (terms[0] - terms[1] - terms[2])[m.free_u]
        assert np.linalg.norm(r) <= 1e-9 * max(np.linalg.norm(t[m.free_u]) for t in terms)
        assert np.all(u1[~m.free_u] == 0) and np.all(p1[~m.free_p] == 0)
        vol = [m.Apu.T @ u1, m.Apu.T @ u0, m.S @ p1, m.S @ p0, dt * (m.C @ p1)]
        r = (vol[0] - vol[1] + vol[2] - vol[3] + vol[4])[m.free_p]
        assert np.linalg.norm(r) <= 1e-8 * max(np.linalg.norm(t[m.free_p]) for t in vol)
        u0, p0 = u1, p1
    a = s.step(prob.dts[6], u.clone(), p.clone(), rtol=1e-10)
    x, y = u.clone(), p.clone()
    s.step(prob.dts[6], u, p, rtol=1e-10)
    s.step(prob.dts[6], x, y, rtol=1e-10)
    assert torch.equal(u, x) and torch.equal(p, y), a      # sums in a fixed order
