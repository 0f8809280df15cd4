"""FP64 products in fixed point: every row within the rounding of FP64 arithmetic, also where
the input is graded over many decades inside a tile, spiky, zero, huge, tiny or not finite.

Bound: an FP64 row sums 8 elements of 24 products through 3 + 3 levels of sums and two
scalings, so its error is at most (24 + 10) eps |A||x| row by row; the same is asked here of
every row (the fixed-point kernel falls back to FP64 arithmetic where it could not hold it).
The parity transform mixes the three fields and eight nodes of an element, so |x| is the
element's largest input."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W
from oracle import fem

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
EPS = 2.0 ** -53

GRIDS = {
    "box_16": dict(nx=16, ny=14, nz=9, shear=(0.0, 0.0)),                    # two tiles in x, one node over
    "dip_ragged": dict(nx=17, ny=3, nz=12, shear=(1.7320508075688772, 0.0), k_perp=1e-13),
    "skew_one_cell": dict(nx=1, ny=1, nz=2, shear=(0.4, -0.3)),
    "box_thin": dict(nx=2, ny=31, nz=2, shear=(0.0, 0.0)),
}
FIELDS = ["noise", "decay", "steep", "spike", "zero", "huge", "tiny", "antisymmetric"]


def field(kind, prob, seed):
    rng = np.random.default_rng(seed)
    N = prob.n_nodes
    n = np.arange(N)
    i, j, k = n % (prob.nx + 1), (n // (prob.nx + 1)) % (prob.ny + 1), n // ((prob.nx + 1) * (prob.ny + 1))
    r = np.sqrt((i - prob.nx / 2) ** 2 + (j - prob.ny / 2) ** 2 + (k - prob.n_planes / 2) ** 2)
    noise = rng.uniform(-1.0, 1.0, (4, N))
    if kind == "noise":
        return noise
    if kind == "decay":
        return np.exp(-r / 3.0) * (1.0 + 0.1 * noise)
    if kind == "steep":
        return np.exp(-r / 0.3) * (1.0 + 0.1 * noise)
    if kind == "spike":
        return (n == N // 2) * (1.0 + 0.1 * noise)
    if kind == "zero":
        return np.zeros((4, N))
    if kind == "huge":
        return 1e250 * noise
    if kind == "tiny":
        return 1e-290 * noise
    return (i - prob.nx / 2) * (1.0 + 1e-3 * noise)


def problem(name, seed=3):
    prob = W.tiny_faulted(seed=seed, h=(0.4, 0.3, 0.5), **GRIDS[name])
    prob.kf = prob.fault = None                        # the bulk blocks alone
    N = prob.n_nodes
    prob.fixed = np.zeros((4, N), np.uint8)
    prob.fixed[0:3, : prob.nx + 1] = 1
    prob.fixed[3, -2:] = 1
    prob.fu, prob.fp = np.zeros((3, N)), np.zeros(N)
    return prob


@pytest.mark.gpu
@pytest.mark.parametrize("kind", FIELDS)
@pytest.mark.parametrize("name", list(GRIDS))
def test_products_within_fp64_rounding_row_by_row(name, kind):
    from gpu_common import cuda, need_gpu, solver_for
    need_gpu()
    prob = problem(name)
    model = fem.Model(prob)
    s = solver_for(prob)
    N = prob.n_nodes
    free = prob.fixed == 0
    x = field(kind, prob, 5) * free
    conn = model.conn
    big = np.zeros(N)                                  # largest input of the elements around a node
    for rows, op in ((x[:3], "KB"), (x[:3], "AUP"), (x[3:], "APU")):
        big[:] = 0.0
        np.maximum.at(big, conn.ravel(), np.repeat(np.abs(rows).max(0)[conn].max(1), 8))
        A = {"KB": model.Kb, "APU": model.Apu, "AUP": model.Apu.T.tocsr()}[op]
        with np.errstate(over="ignore"):
            ref = A @ rows.reshape(-1)
            scale = np.abs(A) @ np.ones(A.shape[1])
        y = s.apply(op, cuda(rows if op != "APU" else rows[0])).cpu().numpy().reshape(-1)
        out = (free[:3] if op != "AUP" else free[3:]).reshape(-1)
        bound = (34 + 34) * EPS * scale * np.tile(big, A.shape[0] // N)    # both sides round
        assert np.all(np.isfinite(y))
        assert np.all(np.abs(y - ref)[out] <= bound[out]), (op, np.max(np.abs(y - ref)[out] / np.maximum(bound[out], 1e-320)))
        assert np.all(y[~out] == 0.0)


CONTRAST = {"even": lambda r, n: np.full(n, 1e-15), "lognormal": lambda r, n: 10.0 ** r.normal(-15.0, 0.5, n),
            "layers": lambda r, n: r.choice([0.0, 1e-19, 1e-12], n), "extreme": lambda r, n: 10.0 ** r.uniform(-40, 0, n),
            "none": lambda r, n: np.zeros(n)}


@pytest.mark.gpu
@pytest.mark.parametrize("dt", [2.0, 1e-9, 1e9])
@pytest.mark.parametrize("kind", ["noise", "decay", "steep", "spike", "zero", "antisymmetric"])
@pytest.mark.parametrize("contrast", list(CONTRAST))
def test_flow_products_within_fp64_rounding_row_by_row(contrast, kind, dt):
    from gpu_common import cuda, need_gpu, solver_for
    need_gpu()
    prob = problem("dip_ragged")
    prob.k = CONTRAST[contrast](np.random.default_rng(9), prob.n_el)
    model = fem.Model(prob)
    s = solver_for(prob)
    s.timestep(dt)
    free = prob.fixed[3] == 0
    p = field(kind, prob, 5)[3] * free
    # element by element: what its own coefficients make of its largest input
    from oracle.fem import element_matrices
    X = model.mesh.coords()[model.conn]
    cond = np.asarray(prob.k) / prob.mu_f
    _, _, S, C = element_matrices(X, prob.E, prob.nu, prob.alpha, 1.0 / prob.M, cond)
    big = np.abs(p)[model.conn].max(1)
    rows = (np.abs(S) + dt * np.abs(C)).sum(2) * big[:, None]
    scale = np.zeros(prob.n_nodes)
    np.add.at(scale, model.conn.ravel(), rows.ravel())
    ref = model.S @ p + dt * (model.C @ p)
    y = s.apply("A22", cuda(p)).cpu().numpy()
    assert np.all(np.abs(y - ref)[free] <= (34 + 34) * EPS * scale[free])
    assert np.all(y[~free] == 0.0)


@pytest.mark.gpu
def test_flow_solves_follow_a_new_permeability():
    from gpu_common import cuda, need_gpu, solver_for
    need_gpu()
    prob = problem("box_16")
    rng = np.random.default_rng(4)
    b = cuda(rng.normal(size=prob.n_nodes) * 1e-12 * (prob.fixed[3] == 0))
    s = solver_for(prob)
    s.timestep(3.0)
    for scale in (1.0, 1e5, 1e-6):
        k = prob.k * scale
        s.set_permeability(k)
        x, _ = s.pcg("A22", b, rtol=1e-12)
        fresh = problem("box_16")
        fresh.k = k
        f = solver_for(fresh)
        f.timestep(3.0)
        y, _ = f.pcg("A22", b, rtol=1e-12)
        assert bool((x == y).all())


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_values_that_are_not_finite_reach_their_rows(bad):
    from gpu_common import cuda, need_gpu, solver_for
    need_gpu()
    prob = problem("box_16")
    model = fem.Model(prob)
    s = solver_for(prob)
    N = prob.n_nodes
    u = field("noise", prob, 6)[:3]
    u[1, N // 2] = bad
    y = s.apply("KB", cuda(u)).cpu().numpy()
    touched = np.zeros(N, bool)
    touched[model.conn[(model.conn == N // 2).any(1)].ravel()] = True
    free = prob.fixed[:3] == 0
    assert np.all(np.isfinite(y[:, ~touched]))
    assert not np.any(np.isfinite(y[1, touched & free[1]]))
    u[1, N // 2] = 0.3
    u[:, prob.fixed[0] == 1] = bad                     # constrained entries are ignored
    assert np.all(np.isfinite(s.apply("KB", cuda(u)).cpu().numpy()))


HOST = r"""
#include <cmath>
#define __host__
#define __device__
#include "gm_fixed.cuh"
extern "C" {
void from_double(double x, int top, int* l) { int v[3]; gm_fx_from_double(x, top, v); for (int i = 0; i < 3; ++i) l[i] = v[i]; }
void coef(double x, int top, int* l) { int v[3]; gm_fx_coef(x, top, v); for (int i = 0; i < 3; ++i) l[i] = v[i]; }
void coef22(double x, int top, int* l) { int v[3]; gm_fx_coef22(x, top, v); for (int i = 0; i < 3; ++i) l[i] = v[i]; }
void product2(const int* x, const int* k, int n, int* l)
{
    FxAcc s{0, 0, 0};
    for (int i = 0; i < n; ++i) { int v[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]}; gm_fx_mac2(s, v, k[2 * i + 1], k[2 * i]); }
    int r[3];
    gm_fx_carry(s, r);
    for (int i = 0; i < 3; ++i) l[i] = r[i];
}
double to_double(int a, int b, int c) { return gm_fx_to_double(a, b, c); }
double to_double4(int a, int b, int c, int d) { return gm_fx_to_double4(a, b, c, d); }
void product4(const int* x, const int* k, int n, int* l)
{
    FxAcc4 s{0, 0, 0, 0};
    for (int i = 0; i < n; ++i) { int v[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]}; gm_fx_mac4(s, v, k[3 * i + 2], k[3 * i + 1], k[3 * i]); }
    int r[4];
    gm_fx_carry4_signed(s, r);
    for (int i = 0; i < 4; ++i) l[i] = r[i];
}
void product(const int* x, const int* k, int n, int sgn, int* l)
{
    FxAcc s{0, 0, 0};
    for (int i = 0; i < n; ++i) { int v[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]}; gm_fx_mac(s, v, k[3 * i + 2], k[3 * i + 1], k[3 * i]); }
    int r[3];
    if (sgn) gm_fx_carry_signed(s, r); else gm_fx_carry(s, r);
    for (int i = 0; i < 3; ++i) l[i] = r[i];
}
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("fixed")
    (d / "h.cpp").write_text(HOST)
    so = str(d / "h.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2410_17133_gb300", "csrc"), "-o", so, str(d / "h.cpp")], check=True)
    lib = ctypes.CDLL(so)
    lib.to_double.restype = lib.to_double4.restype = ctypes.c_double
    lib.from_double.argtypes = lib.coef.argtypes = lib.coef22.argtypes = [ctypes.c_double, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    return lib


def value(l):
    return (int(l[2]) << 52) + (int(l[1]) << 26) + int(l[0])


def test_limbs_and_back(host):
    rng = np.random.default_rng(1)
    l = (ctypes.c_int * 3)()
    for x in [0.0, 5e-324, 2.0 ** -75, -(2.0 ** -75), 0.5, -0.999999999999999889, 2.0 ** -23] + list(
            rng.uniform(-1, 1, 500) * 2.0 ** -rng.integers(0, 90, 500).astype(float)):
        host.from_double(x, 1022, l)
        m, e = float(x).as_integer_ratio()
        exact = (abs(m) << 75) // e
        assert value(l) == (exact if x >= 0 else -exact)
        host.coef(abs(x), 1022, l)
        assert value(l) == (abs(m) << 78) // e
    for _ in range(500):
        a, b = (int(v) for v in rng.integers(-2 ** 31 + 1, 2 ** 31, 2) >> rng.integers(0, 31, 2))
        c = int(rng.integers(-2 ** 30, 2 ** 30)) >> int(rng.integers(0, 31))
        assert host.to_double(a, b, c) == float((c << 52) + (b << 26) + a)   # int -> float rounds to nearest even


def test_two_limb_coefficients(host):
    rng = np.random.default_rng(8)
    l = (ctypes.c_int * 3)()
    P = ctypes.POINTER(ctypes.c_int)
    for t in range(300):
        c = float(rng.uniform(0, 1)) * 2.0 ** -int(rng.integers(0, 90))
        host.coef22(c, 1022, l)
        m, e = c.as_integer_ratio()
        assert (int(l[2]) << 52) + (int(l[1]) << 26) + int(l[0]) == (m << 74) // e
        # a row of entries whose absolute sum is 1, at the largest inputs, on one sign or mixed
        n = int(rng.integers(1, 25))
        w = rng.dirichlet(np.ones(n)) if t % 2 else np.eye(n)[0]
        s = np.ones(n, int) if t % 4 < 2 else rng.choice([-1, 1], n)
        k = np.zeros((n, 2), np.int32)
        x = np.zeros((n, 3), np.int32)
        for i in range(n):
            v = int(w[i] * 2 ** 56) * int(s[i])
            hi = (v + 2 ** 25) >> 26
            k[i] = [v - (hi << 26), hi]
            x[i] = int(s[i]) * np.array([2 ** 29 - 8, 2 ** 29 - 8, 2 ** 26 - 8])
        host.product2(x.ctypes.data_as(P), k.ctypes.data_as(P), n, l)
        exact = sum(value(x[i]) * ((int(k[i][1]) << 26) + int(k[i][0])) for i in range(n))
        # limbs weigh 2^48, 2^22, 2^-4; the pair left out is below 2^54 2^-56
        assert abs(value(l) * 2 ** 52 - exact) <= (2 + 16 * n) * 2 ** 52


def test_four_limbs_and_back(host):
    from fractions import Fraction
    rng = np.random.default_rng(7)
    for t in range(2000):
        a, b, c = (int(v) for v in rng.integers(-2 ** 30, 2 ** 30, 3) >> rng.integers(0, 31, 3))
        d = int(rng.integers(-2 ** 29, 2 ** 29)) >> int(rng.integers(0, 30))
        if t % 3 == 0:
            d = 0 if t % 2 else -1                     # cancelling parts of either sign
        v = Fraction((d << 52) + (c << 26) + b) + Fraction(a, 2 ** 26)
        y = host.to_double4(a, b, c, d)
        assert abs(Fraction(y) - v) <= abs(v) * Fraction(1, 2 ** 52)
    out = (ctypes.c_int * 4)()
    P = ctypes.POINTER(ctypes.c_int)
    for _ in range(300):
        n = int(rng.integers(1, 4))
        x = np.ascontiguousarray(rng.integers(-2 ** 29, 2 ** 29, (n, 3)) // [1, 1, 8], dtype=np.int32)
        k = np.ascontiguousarray(rng.integers(-2 ** 24, 2 ** 24, (n, 3)), dtype=np.int32)
        host.product4(x.ctypes.data_as(P), k.ctypes.data_as(P), n, out)
        exact = sum(value(x[i]) * value(k[i]) for i in range(n))
        got = (value(out[1:]) << 26) + int(out[0])     # units of 2^-26
        assert abs(got * 2 ** 52 - exact) <= (2 + 4 * n) * 2 ** 52
        assert all(-2 ** 25 <= out[i] < 2 ** 25 for i in range(3))


@pytest.mark.parametrize("signed", [0, 1])
def test_product_sums_hold_at_the_largest_values(host, signed):
    # 24 terms at the limits: modes of eight inputs of 75 bits, coefficients whose absolute sum is 1
    rng = np.random.default_rng(2)
    for trial in range(200):
        n = int(rng.integers(1, 25))
        k = np.zeros((n, 3), np.int32)
        x = np.zeros((n, 3), np.int32)
        w = rng.dirichlet(np.ones(n)) if trial % 2 else np.eye(n)[0]
        for i in range(n):
            s = 1 if trial % 4 < 2 else int(rng.choice([-1, 1]))
            c = int(w[i] * 2 ** 78) * s
            k[i] = [s * (abs(c) & (2 ** 26 - 1)), s * ((abs(c) >> 26) & (2 ** 26 - 1)), s * (abs(c) >> 52)]
            x[i] = s * np.array([2 ** 29 - 8, 2 ** 29 - 8, 2 ** 26 - 8])
        out = (ctypes.c_int * 3)()
        P = ctypes.POINTER(ctypes.c_int)
        xc, kc = np.ascontiguousarray(x), np.ascontiguousarray(k)
        host.product(xc.ctypes.data_as(P), kc.ctypes.data_as(P), n, signed, out)
        exact = sum(value(x[i]) * value(k[i]) for i in range(n))
        err = (value(out) * 2 ** 78 - exact) / 2 ** 78
        assert abs(err) <= 2 + 16 * n                  # dropped limb pairs: below 2^55 2^-52 each, and two carries
        lim = 2 ** 25 if signed else 2 ** 26
        assert -lim <= out[0] < lim and -lim <= out[1] < lim
