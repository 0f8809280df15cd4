"""The tetrahedral products and steps without assembled rows: the element walk, which meshes too
large for their rows take, on every mesh of test_gpu_tet_rows and in the steps.

Products: bounds of test_gpu_tet_rows.  Steps: K to 1e-12 of its right-hand side and the pressure
system to 1e-10 of its first residual on both routes, times the condition of the systems (1e4 at
most): 1e-7 of the fields.  Newton with the fault stops at 1e-10 on both, times the same: 1e-5."""
import numpy as np
import pytest

import workloads as W
from test_gpu_tet_rows import MESHES, check

from gpu_common import cuda, need_gpu, rel, torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def walk(monkeypatch):
    return lambda on: monkeypatch.setenv("GM_TET_ROWS", "0" if on else "1")


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-12), (torch.float32, 2e-5)])
@pytest.mark.parametrize("name", list(MESHES))
def test_walk_matches_the_assembled_operators(name, dtype, tol, walk):
    need_gpu()
    import paper_2410_17133_gb300 as gm
    walk(True)
    prob = MESHES[name]()
    check(gm.TetSolver.from_problem(prob), prob, dtype, tol)


def test_the_variable_chooses_the_route(walk):
    need_gpu()
    import paper_2410_17133_gb300 as gm
    prob = MESHES["octant5"]()
    x = cuda(np.random.default_rng(2).normal(size=(3, len(prob.nodes))))
    y = []
    for on in (False, True):
        walk(on)
        y.append(gm.TetSolver.from_problem(prob).apply("KB", x, dt=1.0))
    assert not torch.equal(*y) and rel(y[0].cpu(), y[1].cpu()) < 1e-13     # other sums, other roundings


def test_steps_agree_on_both_routes(walk):
    need_gpu()
    import paper_2410_17133_gb300 as gm
    out = []
    for on in (False, True):
        walk(on)
        prob = W.cryer_octant(n=5, steps=10)
        s = gm.TetSolver.from_problem(prob)
        u = torch.zeros((3, s.N), dtype=torch.float64, device="cuda")
        p = torch.zeros(s.N, dtype=torch.float64, device="cuda")
        for dt in prob.dts[4:6]:
            s.step(dt, u, p, rtol=1e-10)
        out.append((u.cpu(), p.cpu()))
    assert rel(out[1][0], out[0][0]) < 1e-7 and rel(out[1][1], out[0][1]) < 1e-7


@pytest.mark.parametrize("precision", [0, 1])
def test_fault_steps_agree_on_both_routes(walk, precision):
    need_gpu()
    import paper_2410_17133_gb300 as gm
    out = []
    for on in (False, True):
        walk(on)
        prob = W.tetrahedralize(W.tiny_faulted(3, 3, 2, Q=2e-4, steps=1))
        s = gm.TetFaultSolver.from_problem(prob)
        u = torch.zeros((3, s.N), dtype=torch.float64, device="cuda")
        p = torch.zeros(s.N, dtype=torch.float64, device="cuda")
        s.fault_step(prob.dts[0], u, p, newton_rtol=1e-10, precision=precision)
        out.append((u.cpu(), p.cpu()))
    assert rel(out[1][0], out[0][0]) < 1e-5 and rel(out[1][1], out[0][1]) < 1e-5
