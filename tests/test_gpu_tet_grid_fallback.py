"""The tetrahedral K solve when its blocks' waits run out: the solve of two launches per iteration
takes over, in the same call, and the context stays usable."""
import pytest

import workloads as W

from gpu_common import need_gpu, rel, torch

pytestmark = pytest.mark.gpu


def fields(monkeypatch, n, **env):
    import paper_2410_17133_gb300 as gm
    for k in ("GM_TET_GRID", "GM_TET_GRID_POLLS"):
        monkeypatch.delenv(k, raising=False)
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    prob = W.cryer_octant(n=n, steps=10)
    s = gm.TetSolver.from_problem(prob)
    u = torch.zeros((3, s.N), dtype=torch.float64, device="cuda")
    p = torch.zeros(s.N, dtype=torch.float64, device="cuda")
    its = [s.step(dt, u, p, rtol=1e-10)["iterations"] for dt in prob.dts[4:6]]
    return u, p, its


@pytest.mark.parametrize("n", [1, 4, 13])
def test_a_wait_that_runs_out_leaves_the_solve_to_the_launches(n, monkeypatch):
    """No poll at all, so that every wait runs out: the fields are those of the launches, bit for bit.
    A mesh read afterwards solves in one launch again (K to 1e-12 on both routes, conditions of 1e4)."""
    need_gpu()
    u0, p0, i0 = fields(monkeypatch, n, GM_TET_GRID="0")
    u1, p1, i1 = fields(monkeypatch, n, GM_TET_GRID_POLLS="0")
    assert torch.equal(u0, u1) and torch.equal(p0, p1) and i0 == i1
    u2, p2, _ = fields(monkeypatch, n)
    assert rel(u2.cpu(), u0.cpu()) < 1e-7 and rel(p2.cpu(), p0.cpu()) < 1e-7
