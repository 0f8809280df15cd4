"""Assembled rows of the tetrahedral operators on meshes whose rows are unlike those of a
regular mesh, against the oracle's matrices: a fan (two nodes in 90 elements), one
tetrahedron, nodes in no element, several meshes and materials in one context.

Bound as in test_gpu_tet: FP64 1e-12, FP32 2e-5 relative to the result's norm."""
import numpy as np
import pytest

import workloads as W
from oracle import tet

from gpu_common import cuda, need_gpu, rel, torch

pytestmark = pytest.mark.gpu


def problem(nodes, tets, E=20e9, k=1e-15):
    nodes, tets = np.asarray(nodes, float), np.asarray(tets)
    e = nodes[tets]
    bad = np.einsum("ij,ij->i", np.cross(e[:, 1] - e[:, 0], e[:, 2] - e[:, 0]), e[:, 3] - e[:, 0]) < 0
    tets[bad, 1], tets[bad, 2] = tets[bad, 2].copy(), tets[bad, 1].copy()
    return W.TetProblem(name="t", nodes=nodes, tets=tets, E=E, nu=0.25, alpha=0.8, M=50e9, k=k, mu_f=1e-3,
                        fixed=np.zeros((4, len(nodes)), np.uint8), load_tris=np.zeros((0, 3), int), sigma0=0.0, dts=[1.0])


def fan(n=90):
    a = np.linspace(0, 2 * np.pi, n, endpoint=False)
    nodes = [[0, 0, -1], [0, 0, 1.2]] + [[np.cos(t), np.sin(t), 0.1 * np.sin(3 * t)] for t in a]
    return problem(nodes, [[0, 1, 2 + i, 2 + (i + 1) % n] for i in range(n)])


def one():
    return problem([[0, 0, 0], [1, 0.1, 0], [0, 1.3, 0.2], [0.1, 0, 0.9]], [[0, 1, 2, 3]])


def loose_nodes():
    p = one()
    nodes = np.concatenate([[[5.0, 5, 5]], p.nodes, [[7.0, 7, 7]]])
    return problem(nodes, p.tets + 1)


MESHES = {"fan": fan, "one": one, "loose_nodes": loose_nodes, "octant5": lambda: W.cryer_octant(n=5, steps=2)}


def check(s, prob, dtype, tol, seed=4, dt=3.0):
    m = tet.TetModel(prob)
    rng = np.random.default_rng(seed)
    u, p = rng.normal(size=(3, m.N)) * 1e-4, rng.normal(size=m.N) * 1e6
    ku, ap = m.Kb @ u.reshape(-1), m.Apu @ p
    au, sp = m.Apu.T @ u.reshape(-1), m.S @ p + dt * (m.C @ p)
    for op, x, ref in (("KB", u, ku), ("APU", p, ap), ("AUP", u, au), ("A22", p, sp)):
        y = s.apply(op, cuda(x, dtype), dt=dt).double().cpu().numpy().reshape(-1)
        assert rel(y, ref) < tol, (op, rel(y, ref))
    y = s.apply("J", cuda(np.concatenate([u, p[None]]), dtype), dt=dt).double().cpu().numpy()
    assert rel(y[:3].reshape(-1), ku - ap) < tol and rel(y[3], au + sp) < tol


@pytest.mark.parametrize("dtype,tol", [(torch.float64, 1e-12), (torch.float32, 2e-5)])
@pytest.mark.parametrize("name", list(MESHES))
def test_rows_match_the_assembled_operators(name, dtype, tol):
    need_gpu()
    import paper_2410_17133_gb300 as gm
    prob = MESHES[name]()
    check(gm.TetSolver.from_problem(prob), prob, dtype, tol)


def test_rows_follow_mesh_and_materials():
    need_gpu()
    import paper_2410_17133_gb300 as gm
    s = gm.TetSolver(0)
    for prob, E, k in ((fan(), 20e9, 1e-15), (fan(), 7e9, 3e-14), (W.cryer_octant(n=4, steps=2), 7e9, 3e-14)):
        s.mesh(prob.nodes, prob.tets)
        s.materials(E, prob.nu, prob.alpha, prob.M, k, prob.mu_f)
        prob.E, prob.k = E, k
        check(s, prob, torch.float64, 1e-12)
    s.materials(11e9, prob.nu, prob.alpha, prob.M, 2e-15, prob.mu_f)     # same mesh, other materials
    prob.E, prob.k = 11e9, 2e-15
    check(s, prob, torch.float64, 1e-12)
    other = one()
    s.mesh(other.nodes, other.tets)                                      # other mesh, materials kept
    other.E, other.k = 11e9, 2e-15
    check(s, other, torch.float64, 1e-12)
