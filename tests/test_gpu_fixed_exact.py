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
    entries that vanish but for rounding: K (field, mode, field, mode), A_up (mode, field, mode),
    |S| (M = 1) and |C| (k/mu = 1)."""
    h, s = np.asarray(prob.h), prob.shear
    a = np.arange(8)
    X = np.stack([(a & 1) * h[0], (a >> 1 & 1) * h[1], (a >> 2) * h[2] + s[0] * (a & 1) * h[0] + s[1] * (a >> 1 & 1) * h[1]], 1)
    K, A, S, C = (np.asarray(m)[0] for m in element_matrices(X[None], np.ones(1), prob.nu, prob.alpha, 1.0, np.ones(1)))
    perm = np.arange(24).reshape(8, 3).T                    # (field, node) of node-major rows
    K = np.einsum("sa,catb,ub->cstu", SIGN, K[perm][:, :, perm], SIGN) / 64.0
    A = np.einsum("sa,cat,ut->ucs", SIGN, A[perm], SIGN) / 64.0
    S, C = (np.abs(SIGN @ m @ SIGN.T) / 64.0 for m in (S, C))
    for M in (K, A, S, C):
        M[np.abs(M) < 1e-12 * np.abs(M).max()] = 0.0
    return K, A, S, C


def compare(op, prob, u, keep, dt=3.0):
    """Both arithmetics on u ((3, N), for J (4, N), for A22 (1, N)), on the nodes `keep` that no
    element of node 0 touches.  The modes of u are exact in FP64."""
    s = solver_for(prob)
    s.timestep(dt)
    conn = connectivity()
    forced = u.copy()
    forced[:, 0] = 1e-30
    shape = {"KB": (3, -1), "AUP": (3, -1), "J": (4, -1), "A22": (-1,)}[op]
    y, z = (s.apply(op, cuda(x.reshape(shape))).cpu().numpy().reshape(-1, prob.n_nodes) for x in (u, forced))
    K, A, S, C = modal(prob)
    x = np.abs(np.einsum("sa,cea->ces", SIGN, u[:, conn]))  # field, element, mode
    flow = lambda p: np.einsum("us,es->eu", S / prob.M, p).sum(1) + dt * prob.k / prob.mu_f * np.einsum(
        "us,es->eu", C, p).sum(1)
    t = []
    if op in ("KB", "J"):
        t = list(prob.E * np.einsum("cstu,teu->ces", np.abs(K), x[:3]).sum(2))
    if op == "J":
        t = [f + np.einsum("ucs,eu->ces", np.abs(A), x[3])[c].sum(1) for c, f in enumerate(t)]
    if op in ("AUP", "J"):
        t.append(np.einsum("ucs,ces->eu", np.abs(A), x[:3]).sum(1) + (flow(x[3]) if op == "J" else 0.0))
    if op == "A22":
        t.append(flow(x[0]))
    scale = np.zeros_like(y)
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


def fields():
    """Large parts that exert no force beside small ones, all with modes that FP64 holds exactly."""
    i, j, k = nodes()
    rng = np.random.default_rng(7)
    noise = rng.integers(-8, 9, (3, i.size)).astype(float)
    one = np.ones_like(i, float)
    tiny = 2.0 ** -27
    return {
        "constant_beside_noise": np.stack([one, tiny * noise[1], tiny * noise[2]]),
        "constant_beside_less": np.stack([one, tiny ** 1.25 * noise[1], 2.0 ** -34 * noise[2]]),
        "translation_and_strain": np.stack([one + tiny * i, 2.0 * one + tiny * k, -one + tiny * (j + 2.0 * i)]),
        "shear_beside_noise": np.stack([one * k, tiny * noise[1], 0.0 * one]),
        "rotation_and_noise": np.stack([-one * j, one * i, 0.0 * one]) + 2.0 ** -30 * noise,
        "truncated_zero": np.stack([one, 2.0 ** -80 * noise[1], 0.0 * one]),
        "one_component": np.stack([0.0 * one, 0.0 * one, noise[2]]),
    }


@pytest.mark.parametrize("name", list(fields()))
@pytest.mark.parametrize("op", ["KB", "AUP", "J"])
@pytest.mark.parametrize("cell", ["cube", "dip", "flat10", "flat_skew"])
def test_large_parts_without_force_take_no_bits_from_small_ones(cell, op, name, monkeypatch):
    need_gpu()
    prob = problem(cell, monkeypatch)
    k = nodes()[2]
    u = np.where(k >= 3, fields()[name], 0.0)
    if op == "J":
        u = np.concatenate([u, np.where(k >= 3, 1e3 * (1.0 + 2.0 ** -30 * k), 0.0)[None]])
    compare(op, prob, u, k >= 5)


@pytest.mark.parametrize("op", ["KB", "J"])
@pytest.mark.parametrize("above", [0.0, 1.0])
@pytest.mark.parametrize("size", [2.0 ** -1040, 2.0 ** -1046])
def test_subnormal_fields_exert_their_forces(size, above, op, monkeypatch):
    """Multiples of a subnormal, alone and with ones in the planes below: the stiffness carries their
    forces into the normal range."""
    need_gpu()
    prob = problem("cube", monkeypatch)
    k = nodes()[2]
    noise = size * np.random.default_rng(7).integers(-8, 9, (3, k.size))
    u = np.where(k >= 8, noise, np.where((k >= 3) & (k <= 6), above, 0.0))
    if op == "J":
        u = np.concatenate([u, np.zeros((1, k.size))])
    compare(op, prob, u, k >= 9)


@pytest.mark.parametrize("direction", [0, 1, 2])
@pytest.mark.parametrize("dt", [1e-3, 1e3, 1e8])
@pytest.mark.parametrize("cell", ["cube", "dip", "flat100"])
def test_small_pressure_gradients_on_a_large_mean(cell, dt, direction, monkeypatch):
    need_gpu()
    prob = problem(cell, monkeypatch)
    ijk = nodes()
    p = np.where(ijk[2] >= 3, 1.0 + 2.0 ** -26 * ijk[direction], 0.0)[None]
    compare("A22", prob, p, ijk[2] >= 5, dt=dt)


def test_solves_on_flat_cells_where_tiles_change_their_arithmetic(monkeypatch):
    """PCG whose products (with their dot products) start over in FP64: the residual meets the
    tolerance, recomputed by the product."""
    need_gpu()
    prob = problem("flat100", monkeypatch)
    i, j, k = nodes()
    prob.fixed[:3, k == 0] = 1
    s = solver_for(prob)
    s.set_preconditioner(0)
    u = np.stack([1.0 + 2.0 ** -20 * i, 2.0 ** -22 * j, 2.0 ** -24 * (i + k)]) * (prob.fixed[:3] == 0)
    import torch
    b = s.apply("KB", cuda(u))
    x, rep = s.pcg("KT", b, rtol=1e-8)
    assert torch.linalg.norm(b - s.apply("KB", x)) <= 1e-7 * torch.linalg.norm(b), rep
