"""FP64 products in fixed point against the FP64 arithmetic that they stand for, term by term.

A value of 1e-30 at a far corner grades the tile beyond what fixed point takes, so the same
product then runs in FP64 arithmetic with the same entries.  At nodes whose elements the corner
does not touch both must agree within the rounding of the terms that are there: an FP64 row sums
8 elements of 24 products through 3 + 3 levels of sums and two scalings, so each side is within
34 eps of the sum of |entry| |mode| (the fixed-point side is asked to be no worse)."""
import numpy as np
import pytest

import workloads as W
from oracle.fem import element_matrices

from gpu_common import cuda, need_gpu, solver_for

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
NX, NY, NZ = 6, 5, 12
SIGN = np.array([[(-1.0) ** bin(s & a).count("1") for a in range(8)] for s in range(8)])

CELLS = {  # h, shear, nu
    "cube": ((1.0, 1.0, 1.0), (0.0, 0.0), 0.25), "stiff": ((1.0, 1.0, 1.0), (0.0, 0.0), 0.49),
    "flat10": ((10.0, 10.0, 1.0), (0.0, 0.0), 0.25), "flat100": ((100.0, 100.0, 1.0), (0.0, 0.0), 0.25),
    "flat1000": ((1000.0, 1000.0, 1.0), (0.0, 0.0), 0.25), "strip": ((1 / 6, 1 / 200, 1 / 6), (0.0, 0.0), 0.25),
    "dip": ((1.0, 1.0, 1.0), (1.7320508075688772, 0.0), 0.25), "flat_skew": ((30.0, 20.0, 1.0), (0.02, -0.03), 0.3)}


def problem(cell, monkeypatch):
    monkeypatch.setenv("GM_BULK_ZCHUNK", str(NZ + 1))       # one tile
    h, shear, nu = CELLS[cell]
    prob = W.tiny_faulted(NX, NY, NZ, seed=3, h=h, shear=shear)
    prob.kf = prob.fault = None
    prob.nu = nu
    N = prob.n_nodes
    prob.E = np.random.default_rng(1).uniform(1e10, 2e10, prob.n_el)
    prob.fixed = np.zeros((4, N), np.uint8)
    prob.fu, prob.fp = np.zeros((3, N)), np.zeros(N)
    return prob


def nodes():
    n = np.arange((NX + 1) * (NY + 1) * (NZ + 1))
    return n % (NX + 1), (n // (NX + 1)) % (NY + 1), n // ((NX + 1) * (NY + 1))


def connectivity():
    i, j, k = nodes()
    low = np.flatnonzero((i < NX) & (j < NY) & (k < NZ))
    return np.stack([low + (a & 1) + (NX + 1) * ((a >> 1) & 1) + (NX + 1) * (NY + 1) * (a >> 2) for a in range(8)], 1)


def modal(prob):
    """Element blocks of one cell (E = 1) in the basis of the element's parity modes, without the
    entries that vanish but for rounding: K (field, mode, field, mode), A_up (mode, field, mode)."""
    h, s = np.asarray(prob.h), prob.shear
    a = np.arange(8)
    X = np.stack([(a & 1) * h[0], (a >> 1 & 1) * h[1], (a >> 2) * h[2] + s[0] * (a & 1) * h[0] + s[1] * (a >> 1 & 1) * h[1]], 1)
    K, A, _, _ = element_matrices(X[None], np.ones(1), prob.nu, prob.alpha, 1.0, np.ones(1))
    K, A = np.asarray(K)[0], np.asarray(A)[0]
    perm = np.arange(24).reshape(8, 3).T                    # (field, node) of node-major rows
    K = np.einsum("sa,catb,ub->cstu", SIGN, K[perm][:, :, perm], SIGN) / 64.0
    A = np.einsum("sa,cat,ut->ucs", SIGN, A[perm], SIGN) / 64.0
    for M in (K, A):
        M[np.abs(M) < 1e-12 * np.abs(M).max()] = 0.0
    return K, A


def compare(op, prob, u, keep):
    """Both arithmetics on u (3, N), on the nodes `keep` that no element of node 0 touches."""
    s = solver_for(prob)
    conn = connectivity()
    forced = u.copy()
    forced[:, 0] = 1e-30
    y, z = (s.apply(op, cuda(x)).cpu().numpy().reshape(-1, prob.n_nodes) for x in (u, forced))
    K, A = modal(prob)
    x = np.abs(np.einsum("sa,cea->ces", SIGN, u[:, conn]))  # field, element, mode
    scale = np.zeros_like(y)
    if op == "KB":
        t = prob.E * np.einsum("cstu,teu->ces", np.abs(K), x).sum(2)
    else:
        t = np.einsum("ucs,ces->eu", np.abs(A), x).sum(1)[None]
    for c in range(len(scale)):
        np.add.at(scale[c], conn.ravel(), np.repeat(t[c], 8))
    err = np.abs(y - z)[:, keep]
    bound = 34 * EPS * scale[:, keep]
    assert np.all(err <= bound), float((err / np.where(bound > 0, bound, 1e-300)).max())


@pytest.mark.parametrize("direction", [0, 1, 2])
@pytest.mark.parametrize("component", [0, 1, 2])
@pytest.mark.parametrize("op", ["KB", "AUP"])
@pytest.mark.parametrize("cell", list(CELLS))
def test_stretches_and_shears_one_at_a_time(cell, op, component, direction, monkeypatch):
    need_gpu()
    prob = problem(cell, monkeypatch)
    ijk = nodes()
    u = np.zeros((3, prob.n_nodes))
    u[component] = np.where(ijk[2] >= 3, 1.0 + ijk[direction], 0.0)
    compare(op, prob, u, ijk[2] >= 5)
