"""What is measured: the calls that a program built on this framework spends its time in.

A case is one pass through public entry points of ``paper_2410_17133_gb300``: operator
products of a Krylov method of the caller's own, the Newton residual with the fault law,
an inner solve, whole implicit steps from a restored checkpoint, the gradient of a step,
and the same on tetrahedra.  ``listed()`` names the cases, ``draw()`` gives more of the
same ranges, ``exact()`` computes what a pass returns with plain torch in 64 bits.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2410_17133_gb300 as gm

DEV = "cuda"
F64 = torch.float64
MU_F, ALPHA, M_BIOT, NU = 1e-3, 0.8, 50e9, 0.25
TAN60 = math.tan(math.radians(60.0))
# affine cells: an upright box, a fault that dips 60 degrees, a cell sheared both ways
SHEAR = {"box": (0.0, 0.0), "dip": (TAN60, 0.0), "skew": (0.18, -0.1)}
GAUSS = 1.0 / math.sqrt(3.0)


def listed():
    return [
        # the smallest grid: a product of a few microseconds, where launches count
        dict(name="products_f64_8", kind="products", ops="J", nx=8, ny=8, nz=8, cell="box", k_perp=0.0, dtype="f64"),
        # every operator once, in single precision, on the 160^3 grid with a dipping fault
        dict(name="products_f32_160", kind="products", ops="KT,APU,AUP,A22,J", nx=160, ny=160, nz=160, cell="dip",
             k_perp=0.0, dtype="f32"),
        # the stiffness product in double precision on a large grid
        dict(name="stiffness_f64_128", kind="products", ops="KT", nx=128, ny=128, nz=128, cell="dip", k_perp=0.0,
             dtype="f64"),
        # the four blocks of a partitioned solve in double precision: ragged sizes, a cell
        # sheared both ways, lips with pressures of their own
        dict(name="blocks_f64_ragged", kind="products", ops="KT,APU,AUP,A22", nx=61, ny=127, nz=46, cell="skew",
             k_perp=1e-18, dtype="f64"),
        # return map and Newton residual, once per Newton iteration of every step
        dict(name="residual_f64_64", kind="residual", nx=64, ny=64, nz=64, cell="box", k_perp=0.0),
        # one displacement solve in double precision to a tight tolerance
        dict(name="solve_kt_f64_48", kind="solve", which="KT", nx=48, ny=48, nz=48, cell="dip", k_perp=0.0, rtol=1e-12),
        # the whole run of the unit cube with 8^3 cells: five steps in double precision, inexact inner solves
        dict(name="run_f64_8", kind="run", nx=8, ny=8, nz=8, cell="box", k_perp=0.0, dtype="f64", steps=5, dt=2.0,
             Q=5e-5, uniform=True, rtol=1e-12),
        # one step of the 64^3 log-normal cube, single-precision inner solves
        dict(name="step_f32_64", kind="run", nx=64, ny=64, nz=64, cell="box", k_perp=0.0, dtype="f32", steps=1, dt=0.1,
             Q=2e-5, uniform=False, rtol=1e-13),
        # one step of the 160^3 grid with the dipping fault, single-precision inner solves
        dict(name="step_f32_160", kind="run", nx=160, ny=160, nz=160, cell="dip", k_perp=0.0, dtype="f32", steps=1,
             dt=5.0, Q=2e-4, uniform=False, rtol=1e-13),
        # gradient of slip and pressure observations of a step (backward of a step)
        dict(name="gradient_32", kind="gradient", nx=32, ny=32, nz=32, cell="box", k_perp=0.0, Q=2e-5, dt=0.1),
        # tetrahedra: the coupled product on the octant mesh of a ball, and one step of Cryer's problem
        dict(name="tet_products_f64_32", kind="tet_products", ops="KB,APU,AUP,A22,J", n=32, dtype="f64"),
        dict(name="tet_step_f64_16", kind="tet_step", n=16, dt_rel=1e-3, rtol=1e-10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["products"] * 5 + ["residual", "solve", "run", "run", "gradient", "tet_products", "tet_step"])
    cell = rng.choice(["box", "dip", "skew"])
    k_perp = rng.choice([0.0, 0.0, 1e-18])
    if kind == "tet_products":
        ops = rng.choice(["KB", "J", "KB,APU,AUP,A22"])
        return dict(kind=kind, ops=ops, n=_log_int(rng, 4, 36), dtype=rng.choice(["f32", "f64"]))
    if kind == "tet_step":
        return dict(kind=kind, n=_log_int(rng, 4, 16), dt_rel=10.0 ** rng.uniform(-4.0, -1.5), rtol=1e-10)
    if kind == "products":
        while True:
            nx, ny, nz = (_log_int(rng, 6, 200) for _ in range(3))
            if nx * ny * nz <= 160 ** 3:
                break
        return dict(kind=kind, ops=rng.choice(["KT", "J", "A22", "APU,AUP", "KB", "KT,APU,AUP,A22", "KT,APU,AUP,A22,J"]),
                    nx=nx, ny=ny, nz=nz, cell=cell, k_perp=k_perp, dtype=rng.choice(["f32", "f64"]))
    if kind == "residual":
        nx, ny, nz = (_log_int(rng, 6, 90) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, cell=cell, k_perp=k_perp)
    if kind == "solve":
        n = [_log_int(rng, 6, 44) for _ in range(3)]
        return dict(kind=kind, which=rng.choice(["KT", "A22"]), nx=n[0], ny=n[1], nz=n[2], cell=rng.choice(["box", "dip"]),
                    k_perp=k_perp, rtol=1e-12)
    if kind == "gradient":
        n = 2 * _log_int(rng, 4, 16)
        return dict(kind=kind, nx=n, ny=n, nz=n, cell="box", k_perp=0.0, Q=2e-5, dt=0.1)
    dtype = rng.choice(["f32", "f32", "f64"])
    n = _log_int(rng, 6, 14 if dtype == "f64" else 44)
    dip = rng.random() < 0.5
    # 1 m cells with the dipping fault, or a unit cube
    return dict(kind="run", nx=n, ny=n + rng.randrange(-1, 2), nz=n + (n % 2 if rng.random() < 0.7 else 1 - n % 2),
                cell="dip" if dip else "box", k_perp=0.0, dtype=dtype, steps=rng.choice([1, 2]), dt=5.0 if dip else 0.1,
                Q=2e-4 if dip else 2e-5, uniform=False, rtol=1e-13)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _grid(case, seed):
    """The problem description that Solver.from_problem takes."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    kf = nz // 2
    nb, npl = (nx + 1) * (ny + 1), nz + 2
    N, nel = nb * npl, nx * ny * nz
    rng = np.random.default_rng(seed)
    h = (1.0, 1.0, 1.0) if case["cell"] == "dip" else (1.0 / nx, 1.0 / ny, 1.0 / nz)
    if case.get("uniform"):
        E, k = np.full(nel, 20e9), np.full(nel, 1e-15)
        strength = rng.uniform(0.95, 1.05)
    else:
        E, k = rng.uniform(10e9, 30e9, nel), 10.0 ** rng.normal(-15.0, 0.5, nel)
        strength = 1.0
    fixed = np.zeros((4, N), np.uint8)
    fixed[0:3, :nb] = 1                                   # bottom face held
    fp = np.zeros(N)
    well = nx // 2 + (nx + 1) * (ny // 2) + nb * kf       # injection at the centre pair, half to each lip
    fp[well] = fp[well + nb] = 0.5 * case.get("Q", 0.0) * strength
    fault = SimpleNamespace(kn=2e12, ks=2e11, f=0.6, w0=1e-4, wk_par=1e-15, k_perp=case["k_perp"], MF=0.2e6, tn0=10e6,
                            tau0=(5.4e6, 0.0))
    return SimpleNamespace(nx=nx, ny=ny, nz=nz, kf=kf, nb=nb, n_planes=npl, N=N, nel=nel, origin=(0.0, 0.0, 0.0), h=h,
                           shear=SHEAR[case["cell"]], fault=fault, E=E, k=k, nu=NU, alpha=ALPHA, M=M_BIOT, mu_f=MU_F,
                           fixed=fixed, fu=np.zeros((3, N)), fp=fp)


def _fields(g, seed):
    """Displacement and pressure as an iteration meets them: smooth modes, a part that decays from the
    well, and noise; jumps over the fault that leave pairs open, sticking and slipping."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rnd = lambda *s: torch.rand(*s, generator=gen, device=DEV, dtype=F64)
    z, y, x = (torch.linspace(0.0, 1.0, n, device=DEV, dtype=F64) for n in (g.n_planes, g.ny + 1, g.nx + 1))
    X, Y, Z = x[None, None, :], y[None, :, None], z[:, None, None]
    near = torch.exp(-4.0 * torch.sqrt((X - 0.5) ** 2 + (Y - 0.5) ** 2 + (Z - 0.5) ** 2 + 1e-4))
    f = torch.empty((4, g.n_planes, g.ny + 1, g.nx + 1), device=DEV, dtype=F64)
    for c in range(4):
        a = (1.0 + 4.0 * rnd(6)).tolist()
        f[c] = torch.sin(a[0] * X + a[1]) * torch.cos(a[2] * Y + a[3]) * torch.sin(a[4] * Z + a[5]) + 2.0 * near
        f[c] += 0.1 * (2.0 * rnd(*f.shape[1:]) - 1.0)
    u, p = 1e-5 * f[:3].reshape(3, g.N), 1e6 * f[3].reshape(g.N)
    lo = slice(g.kf * g.nb, (g.kf + 1) * g.nb)
    up = slice((g.kf + 1) * g.nb, (g.kf + 2) * g.nb)
    u[:, up] = u[:, lo] + 6e-6 * (2.0 * rnd(3, g.nb) - 1.0)
    u *= torch.as_tensor(1 - g.fixed[:3], device=DEV)
    if not g.fault.k_perp > 0:
        p[up] = p[lo]
    return u, p


def _observe(g, seed):
    """Derivatives of an objective that sums slip at some pairs and pressure at some nodes."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 7)
    ds = torch.zeros((2, g.nb), device=DEV, dtype=F64)
    dp = torch.zeros(g.N, device=DEV, dtype=F64)
    pairs = torch.randperm(g.nb, generator=gen, device=DEV)[:min(256, g.nb)]
    nodes = torch.randperm(g.kf * g.nb, generator=gen, device=DEV)[:64]
    ds[0, pairs] = 1e6 * (0.5 + torch.rand(pairs.numel(), generator=gen, device=DEV, dtype=F64))
    dp[nodes] = 1e-6 * (0.5 + torch.rand(nodes.numel(), generator=gen, device=DEV, dtype=F64))
    return dp, ds


def _octant(n):
    """Octant of the unit ball: the unit cube's n^3 cells mapped radially, six Kuhn tetrahedra each."""
    g = np.linspace(0.0, 1.0, n + 1)
    P = np.stack([a.ravel() for a in np.meshgrid(g, g, g, indexing="ij")], 1)
    ninf, n2 = np.abs(P).max(1), np.linalg.norm(P, axis=1)
    nodes = P * np.where(n2 > 0, ninf / np.where(n2 > 0, n2, 1.0), 0.0)[:, None]
    I = np.stack([a.ravel() for a in np.meshgrid(*[np.arange(n)] * 3, indexing="ij")], 1)
    nid = lambda q: (q[:, 0] * (n + 1) + q[:, 1]) * (n + 1) + q[:, 2]
    tets = []
    for path in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        q, ids = I.copy(), [nid(I)]
        for ax in path:
            q[:, ax] += 1
            ids.append(nid(q))
        tets.append(np.stack(ids, 1))
    tets = np.stack(tets, 1).reshape(-1, 4)
    a, b, c, d = (nodes[tets[:, i]] for i in range(4))
    bad = np.einsum("ij,ij->i", np.cross(b - a, c - a), d - a) < 0
    tets[bad, 1], tets[bad, 2] = tets[bad, 2].copy(), tets[bad, 1].copy()
    N = len(nodes)
    fixed = np.zeros((4, N), np.uint8)
    fixed[0:3] = (P == 0.0).T                             # symmetry planes
    fixed[3] = ninf == 1.0                                # drained, loaded sphere
    tris = []
    for f, opp in (((0, 1, 2), 3), ((0, 1, 3), 2), ((0, 2, 3), 1), ((1, 2, 3), 0)):
        t = tets[:, f]
        on = np.any(np.all(P[t] == 1.0, axis=1), axis=1)
        t, o = t[on], tets[on, opp]
        x0 = nodes[t[:, 0]]
        out = np.einsum("ij,ij->i", np.cross(nodes[t[:, 1]] - x0, nodes[t[:, 2]] - x0), x0 - nodes[o])
        t = np.where((out < 0)[:, None], t[:, [0, 2, 1]], t)
        tris.append(t)
    return SimpleNamespace(nodes=nodes, tets=tets, fixed=fixed, load_tris=np.concatenate(tris), N=N, sigma0=1e6, nu=NU,
                           alpha=ALPHA, M=M_BIOT, mu_f=MU_F)


def _ball(case, seed):
    m = _octant(case["n"])
    rng = np.random.default_rng(seed)
    m.E, m.k, m.sigma0 = rng.uniform(10e9, 30e9), 10.0 ** rng.uniform(-15.5, -14.5), rng.uniform(0.5e6, 2e6)
    # dt in units of the consolidation time of the unit ball
    Kv = m.E * (1 - NU) / ((1 + NU) * (1 - 2 * NU))
    m.dt = case.get("dt_rel", 1e-3) * (1.0 / M_BIOT + ALPHA ** 2 / Kv) * MU_F / m.k
    gen = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.as_tensor(m.nodes, device=DEV)
    r = torch.randn((4, m.N), generator=gen, device=DEV, dtype=F64)
    m.u = 1e-5 * (torch.sin(2.0 * x.T) + 0.1 * r[:3])
    m.p = 1e6 * (torch.cos(x.sum(1)) + 0.1 * r[3])
    return m


_IN = {"KB": "u", "KT": "u", "A22": "p", "APU": "p", "AUP": "u", "J": "up"}


def _operand(op, u, p, dtype):
    x = {"u": u, "p": p, "up": torch.cat([u, p[None]])}[_IN[op]]
    return x.to(torch.float32 if dtype == "f32" else F64).contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind.startswith("tet"):
        m = _ball(case, seed)
        s = gm.TetSolver(0)
        s.mesh(m.nodes, m.tets)
        s.materials(m.E, m.nu, m.alpha, m.M, m.k, m.mu_f)
        if kind == "tet_products":
            return SimpleNamespace(kind=kind, s=s, dt=m.dt,
                                   x={op: _operand(op, m.u, m.p, case["dtype"]) for op in case["ops"].split(",")})
        s.dirichlet(m.fixed)
        s.surface_load(m.load_tris, m.sigma0)
        return SimpleNamespace(kind=kind, s=s, dt=m.dt, rtol=case["rtol"], u=torch.zeros((3, m.N), device=DEV, dtype=F64),
                               p=torch.zeros(m.N, device=DEV, dtype=F64))
    g = _grid(case, seed)
    s = gm.Solver.from_problem(g, device=0)
    st = SimpleNamespace(kind=kind, s=s)
    if kind in ("products", "residual", "solve"):
        u, p = _fields(g, seed)
        s.timestep(2.0)
        if kind != "residual":
            s.fault_update(u)                             # the tangent of the current fault states
    if kind == "products":
        st.x = {op: _operand(op, u, p, case["dtype"]) for op in case["ops"].split(",")}
    elif kind == "residual":
        st.u, st.du, st.dp = u, u, p
    elif kind == "solve":
        # a right-hand side that the operator reaches: a force or flow residual of the field
        st.which, st.rtol = case["which"], case["rtol"]
        free = torch.as_tensor(1 - g.fixed, device=DEV, dtype=F64)
        st.b = (1e5 * u * free[:3] if st.which == "KT" else 1e-15 * p * free[3]).contiguous()
        if st.which == "A22" and not g.fault.k_perp > 0:
            st.b[(g.kf + 1) * g.nb:(g.kf + 2) * g.nb] = 0.0
    elif kind == "run":
        # the checkpoint a program resumes from (here the state before injection)
        st.u0, st.p0 = np.zeros((3, g.N)), np.zeros(g.N)
        st.dlie0, st.flags0 = np.zeros((2, g.nb)), np.ones(g.nb, np.int8)
        st.dts = [case["dt"]] * case["steps"]
        # both precisions at the tolerances of an inexact Newton method (Newton refines to its own)
        st.kw = dict(newton_rtol=case["rtol"], precision=gm.F32 if case["dtype"] == "f32" else gm.F64, inner_rtol=1e-2,
                     outer_rtol=1e-1)
    else:
        s.step(case["dt"], newton_rtol=1e-12, precision=gm.F32, schur_precond=1)
        s.set_adjoint_options(gm.F32, 1e-3, 1)
        st.dp, st.ds = _observe(g, seed)
    return st


def run(st):
    s = st.s
    if st.kind == "products":
        return {op: s.apply(op, x) for op, x in st.x.items()}
    if st.kind == "residual":
        law = s.fault_update(st.u)
        b, rhat = s.residual(st.du, st.dp)
        return dict(law=law, b=b, rhat=rhat)
    if st.kind == "solve":
        return s.pcg(st.which, st.b, rtol=st.rtol, maxit=20000)[0]
    if st.kind == "run":
        s.set_state(u=st.u0, p=st.p0, dlie=st.dlie0, flags=st.flags0)
        for dt in st.dts:
            s.step(dt, **st.kw)
        return s.get_state()
    if st.kind == "gradient":
        g_logk, g_f, g_logQ, _ = s.adjoint(dJ_dp=st.dp, dJ_dslip=st.ds, rtol=1e-12)
        return dict(g_logk=g_logk, g_f=g_f, g_logQ=g_logQ)
    if st.kind == "tet_products":
        return {op: s.apply(op, x, dt=st.dt) for op, x in st.x.items()}
    u, p = st.u.clone(), st.p.clone()
    s.step(st.dt, u, p, rtol=st.rtol)
    return dict(u=u, p=p)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

# per element: multiplications and additions of the element operators on 24 displacements and 8 pressures
# (dense Q1 blocks have 576, 192 and 64 entries; in the modes of an affine cell about 73, 16 and 11 remain)
_FLOPS = {"KB": 400, "KT": 400, "A22": 130, "APU": 200, "AUP": 200, "J": 700}
# vectors read and written per node, and element coefficients
_VALUES = {"KB": 7, "KT": 7, "A22": 3, "APU": 4, "AUP": 4, "J": 10}


def work(case):
    kind = case["kind"]
    if kind.startswith("tet"):
        N, M = (case["n"] + 1) ** 3, 6 * case["n"] ** 3
        size = 4 if case.get("dtype") == "f32" else 8
        # vertex ids, gradients and volume of an element; vectors of a node
        one = lambda op: M * (16 + 13 * size) + N * size * (_VALUES[op] - (1 if op in ("KB", "KT") else 0))
        if kind == "tet_products":
            ops = case["ops"].split(",")
            return {"bytes": sum(one(op) for op in ops), "flops": M * 250 * len(ops)}
        # the inputs and outputs once, and one product of each operator
        return {"bytes": one("J") + 8 * N * 8, "flops": M * 250}
    nel = case["nx"] * case["ny"] * case["nz"]
    N = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 2)
    if kind == "products":
        size = 4 if case["dtype"] == "f32" else 8
        ops = case["ops"].split(",")
        return {"bytes": N * size * sum(_VALUES[op] for op in ops), "flops": nel * sum(_FLOPS[op] for op in ops)}
    if kind == "residual":
        # u, du, dp, the state, loads and diagonals in, the residual out
        return {"bytes": N * 8 * (3 + 4 + 4 + 4 + 4 + 4 + 2), "flops": nel * 800}
    # solves and steps: what goes in and comes out once, with one product of the operators for each
    steps = case.get("steps", 1)
    return {"bytes": N * 8 * (8 + 16 * steps), "flops": nel * 800 * steps}


# ---------------------------------------------------------------------------
# The same in 64 bits, with plain torch
# ---------------------------------------------------------------------------

def _shape(pts):
    """Values and reference derivatives of the trilinear functions at pts (q, 3); node a = ax + 2 ay + 4 az."""
    sgn = torch.tensor([[2.0 * ((a >> d) & 1) - 1.0 for d in range(3)] for a in range(8)], dtype=F64)
    f = 0.5 * (1.0 + sgn[None] * pts[:, None, :])
    n = f.prod(2)
    dn = torch.stack([0.5 * sgn[None, :, d] * f[:, :, (d + 1) % 3] * f[:, :, (d + 2) % 3] for d in range(3)], 2)
    return n, dn


def _strain(G):
    """(..., a, 3) gradients -> (..., 6, 3a) strain rows xx yy zz yz xz xy, columns 3 a + c."""
    B = torch.zeros(G.shape[:-2] + (6, G.shape[-2], 3), dtype=G.dtype, device=G.device)
    for i in range(3):
        B[..., i, :, i] = G[..., i]
    for row, (i, j) in ((3, (1, 2)), (4, (0, 2)), (5, (0, 1))):
        B[..., row, :, i] = G[..., j]
        B[..., row, :, j] = G[..., i]
    return B.flatten(-2)


def _hooke(E, nu):
    lam, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    D = torch.zeros((6, 6), dtype=F64)
    D[:3, :3] = lam
    D += torch.diag(torch.tensor([2 * mu] * 3 + [mu] * 3, dtype=F64))
    return D


class _Exact:
    """The coupled problem of a structured grid, element by element."""

    def __init__(self, g, dt):
        self.g, self.dt = g, dt
        h, (sx, sy) = g.h, g.shear
        cell = torch.tensor([[h[0] * ax, h[1] * ay, h[2] * az + sx * h[0] * ax + sy * h[1] * ay]
                             for az in (0, 1) for ay in (0, 1) for ax in (0, 1)], dtype=F64)
        pts = GAUSS * torch.tensor([[x, y, z] for z in (-1.0, 1.0) for y in (-1.0, 1.0) for x in (-1.0, 1.0)], dtype=F64)
        n, dn = _shape(pts)
        J = torch.einsum("ad,qak->qdk", cell, dn)
        w = torch.linalg.det(J)
        G = torch.einsum("qak,qkd->qad", dn, torch.linalg.inv(J))
        B = _strain(G)
        div = B[:, :3].sum(1)
        self.K = torch.einsum("q,qia,ij,qjb->ab", w, B, _hooke(1.0, g.nu), B).to(DEV)
        self.A = (g.alpha * torch.einsum("q,qa,qb->ab", w, div, n)).to(DEV)
        self.S = (torch.einsum("q,qa,qb->ab", w, n, n) / g.M).to(DEV)
        self.C = torch.einsum("q,qad,qbd->ab", w, G, G).to(DEV)
        T = lambda a: torch.as_tensor(a, device=DEV)
        self.E, self.kap = T(np.asarray(g.E, float)), T(np.asarray(g.k, float) / g.mu_f)
        ek, ej, ei = (a.reshape(-1) for a in torch.meshgrid(*(torch.arange(m, device=DEV) for m in (g.nz, g.ny, g.nx)),
                                                            indexing="ij"))
        kb = ek + (ek >= g.kf)
        self.conn = torch.stack([ei + (a & 1) + (g.nx + 1) * (ej + ((a >> 1) & 1)) + g.nb * (kb + (a >> 2))
                                 for a in range(8)], 1)
        self.tied = not g.fault.k_perp > 0
        self.lo, self.up = slice(g.kf * g.nb, (g.kf + 1) * g.nb), slice((g.kf + 1) * g.nb, (g.kf + 2) * g.nb)
        self.free = torch.as_tensor(1 - g.fixed, device=DEV, dtype=F64)
        if self.tied:
            self.free[3, self.up] = 0.0
        # fault frame, pair areas and the Laplacian of a fault quad
        a1, a2 = torch.tensor([h[0], 0, sx * h[0]], dtype=F64), torch.tensor([0, h[1], sy * h[1]], dtype=F64)
        nrm = torch.linalg.cross(a1, a2)
        self.n, area = (nrm / nrm.norm()).to(DEV), nrm.norm().item()
        self.t1 = (a1 / a1.norm()).to(DEV)
        self.t2 = torch.linalg.cross(self.n, self.t1)
        qj, qi = (a.reshape(-1) for a in torch.meshgrid(torch.arange(g.ny, device=DEV), torch.arange(g.nx, device=DEV),
                                                        indexing="ij"))
        self.quad = torch.stack([qi + (b & 1) + (g.nx + 1) * (qj + (b >> 1)) for b in range(4)], 1)
        self.area = torch.zeros(g.nb, device=DEV, dtype=F64).index_add_(
            0, self.quad.reshape(-1), torch.full((self.quad.numel(),), 0.25 * area, device=DEV, dtype=F64))
        metric = torch.stack([a1, a2], 1) * 0.5
        Gi = torch.linalg.inv(metric.T @ metric)
        L = torch.zeros((4, 4), dtype=F64)
        for x in (-GAUSS, GAUSS):
            for y in (-GAUSS, GAUSS):
                d = torch.tensor([[0.25 * sa * (1 + sb * y), 0.25 * sb * (1 + sa * x)]
                                  for sb in (-1.0, 1.0) for sa in (-1.0, 1.0)], dtype=F64)
                L += 0.25 * area * d @ Gi @ d.T
        self.L = L.to(DEV)
        self.D = None

    def elements(self, mat, x, coef, fields, out):
        """Sum over the elements of coef_e mat x_e, in slices that fit."""
        y = torch.zeros((out, self.g.N), device=DEV, dtype=F64)
        step = 1 << 20
        for s in range(0, self.g.nel, step):
            c = self.conn[s:s + step]
            xe = x[:, c].permute(1, 2, 0).reshape(c.shape[0], 8 * fields)
            ye = xe @ mat.T
            if coef is not None:
                ye = ye * coef[s:s + step, None]
            for f in range(out):
                y[f].index_add_(0, c.reshape(-1), ye[:, f::out].reshape(-1))
        return y

    def law(self, u, dlie=None):
        """Contact and friction at every pair (open 0, stick 1, slip 2) and the symmetric tangent."""
        f = self.g.fault
        tau0 = torch.tensor(f.tau0, device=DEV, dtype=F64)
        jump = (u[:, self.up] - u[:, self.lo]).T
        dlie = torch.zeros((self.g.nb, 2), device=DEV, dtype=F64) if dlie is None else dlie
        dn = jump @ self.n
        gs = torch.stack([jump @ self.t1, jump @ self.t2], 1)
        tn = f.tn0 - f.kn * dn
        contact = tn >= 0
        trial = tau0 + f.ks * (gs - dlie)
        size = trial.norm(dim=1)
        tn = torch.where(contact, tn, 0.0)
        over = size - f.f * tn
        slip = contact & (over > 0) & (size > 0)
        stick = contact & ~slip
        tau = torch.where(slip[:, None], trial / size.clamp_min(1e-300)[:, None], 0.0)
        ts = torch.where(slip[:, None], (f.f * tn)[:, None] * tau, torch.where(stick[:, None], trial, 0.0))
        new = torch.where(slip[:, None], dlie + (over / f.ks)[:, None] * tau, dlie)
        Ts = torch.where(stick[:, None], f.ks * (gs - dlie), ts - tau0)
        T = torch.where(contact, f.kn * dn, f.tn0)[:, None] * self.n + Ts[:, :1] * self.t1 + Ts[:, 1:] * self.t2
        tg = tau[:, :1] * self.t1 + tau[:, 1:] * self.t2
        Pt = torch.outer(self.t1, self.t1) + torch.outer(self.t2, self.t2)
        ratio = torch.where(slip, f.f * tn / size.clamp_min(1e-300), torch.where(stick, 1.0, 0.0))
        self.D = f.kn * contact.double()[:, None, None] * torch.outer(self.n, self.n) + f.ks * ratio[:, None, None] * (
            Pt - tg[:, :, None] * tg[:, None, :])
        flags = torch.where(contact, torch.where(slip, 2, 1), 0).to(torch.int8)
        return dict(flags=flags, tn=tn, ts=ts.T, dlie=new.T, T=T.T, gs=gs.T)

    def _mid(self, p):
        return p[self.lo] if self.tied else 0.5 * (p[self.lo] + p[self.up])

    def _put(self, y, mid):
        """A term tested with the mid-plane pressure, to the rows that carry it."""
        if self.tied:
            y[self.lo] += mid
        else:
            y[self.lo] += 0.5 * mid
            y[self.up] += 0.5 * mid

    def expand(self, p):
        if self.tied:
            p = p.clone()
            p[self.up] = p[self.lo]
        return p

    def fold(self, y):
        if self.tied:
            y[self.lo] += y[self.up]
            y[self.up] = 0.0
        return y

    def Kb(self, u):
        return self.elements(self.K, u, self.E, 3, 3)

    def KT(self, u):
        y = self.Kb(u)
        f = self.area * torch.einsum("pij,jp->ip", self.D, u[:, self.up] - u[:, self.lo])
        y[:, self.up] += f
        y[:, self.lo] -= f
        return y

    def Apu(self, p):
        y = self.elements(self.A, self.expand(p)[None], None, 1, 3)
        f = self.n[:, None] * (self.area * self._mid(p))
        y[:, self.up] += f
        y[:, self.lo] -= f
        return y

    def Aup(self, u):
        y = self.fold(self.elements(self.A.T, u, None, 3, 1)[0])
        self._put(y, self.area * (self.n @ (u[:, self.up] - u[:, self.lo])))
        return y

    def Sp(self, p):
        y = self.fold(self.elements(self.S, self.expand(p)[None], None, 1, 1)[0])
        self._put(y, self.area * self.g.fault.w0 / self.g.fault.MF * self._mid(p))
        return y

    def Cp(self, p):
        g, f = self.g, self.g.fault
        y = self.fold(self.elements(self.C, self.expand(p)[None], self.kap, 1, 1)[0])
        q = self._mid(p)[self.quad] @ self.L.T * (f.wk_par / g.mu_f)
        self._put(y, torch.zeros(g.nb, device=DEV, dtype=F64).index_add_(0, self.quad.reshape(-1), q.reshape(-1)))
        if not self.tied:
            t = self.area * (f.k_perp / (g.mu_f * f.w0)) * (p[self.up] - p[self.lo])
            y[self.up] += t
            y[self.lo] -= t
        return y

    def A22(self, p):
        return self.Sp(p) + self.dt * self.Cp(p)

    def apply(self, op, x):
        fu, fp = self.free[:3], self.free[3]
        if op in ("KB", "KT"):
            return fu * (self.Kb(fu * x) if op == "KB" else self.KT(fu * x))
        if op == "A22":
            return fp * self.A22(fp * x)
        if op == "APU":
            return fu * self.Apu(fp * x)
        if op == "AUP":
            return fp * self.Aup(fu * x)
        u, p = fu * x[:3], fp * x[3]
        return torch.cat([fu * (self.KT(u) - self.Apu(p)), (fp * (self.Aup(u) + self.A22(p)))[None]])

    def diagonals(self):
        g = self.g
        dK = torch.zeros((3, g.N), device=DEV, dtype=F64)
        dS, dC = torch.zeros(g.N, device=DEV, dtype=F64), torch.zeros(g.N, device=DEV, dtype=F64)
        for a in range(8):
            c = self.conn[:, a]
            for d in range(3):
                dK[d].index_add_(0, c, self.E * self.K[3 * a + d, 3 * a + d])
            dS.index_add_(0, c, torch.full((g.nel,), self.S[a, a].item(), device=DEV, dtype=F64))
            dC.index_add_(0, c, self.kap * self.C[a, a])
        f = g.fault
        lap = torch.zeros(g.nb, device=DEV, dtype=F64)
        for b in range(4):
            lap.index_add_(0, self.quad[:, b], torch.full((self.quad.shape[0],), (self.L[b, b] * f.wk_par / g.mu_f).item(),
                                                          device=DEV, dtype=F64))
        st = self.area * f.w0 / f.MF
        if self.tied:
            dS[self.lo] += dS[self.up] + st
            dC[self.lo] += dC[self.up] + lap
        else:
            t = self.area * (f.k_perp / (g.mu_f * f.w0))
            for lip in (self.lo, self.up):
                dS[lip] += 0.25 * st
                dC[lip] += 0.25 * lap + t
        return dK, dS + self.dt * dC

    def residual(self, un, pn, du, dp, T):
        """Momentum and flow residuals of a step from (un, pn), constrained rows zero."""
        u, p = un + du, pn + dp
        b1 = -self.Kb(u) + self.Apu(p)
        b1[:, self.up] -= self.area * T
        b1[:, self.lo] += self.area * T
        src = self.fold(torch.as_tensor(self.g.fp, device=DEV).clone())
        b2 = self.dt * (src - self.Cp(p)) - self.Sp(dp) - self.Aup(du)
        return torch.cat([self.free[:3] * b1, (self.free[3] * b2)[None]])


def _cg(apply, b, dinv, rtol, maxit):
    x, r = torch.zeros_like(b), b.clone()
    z = dinv * r
    p, rz, stop = z.clone(), (r * z).sum(), rtol * b.norm()
    for it in range(maxit):
        q = apply(p)
        a = rz / (p * q).sum()
        x += a * p
        r -= a * q
        if it % 20 == 0 and r.norm() <= stop:
            return x
        z = dinv * r
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return None


def _columns(apply, shape, free):
    """The matrix of `apply` on the free entries, for grids of a few hundred nodes."""
    cols = []
    for i in torch.nonzero(free.reshape(-1)).reshape(-1).tolist():
        e = torch.zeros(shape, device=DEV, dtype=F64)
        e.view(-1)[i] = 1.0
        cols.append(apply(e).reshape(-1))
    return torch.stack(cols, 1)


def _exact_run(case, g):
    """Newton with the assembled Jacobian, for grids of a few hundred nodes."""
    m = _Exact(g, case["dt"])
    free = m.free.reshape(-1) > 0
    un, pn = torch.zeros((3, g.N), device=DEV, dtype=F64), torch.zeros(g.N, device=DEV, dtype=F64)
    dlie = torch.zeros((g.nb, 2), device=DEV, dtype=F64)
    m.law(un)
    m.D.zero_()
    J0 = _columns(lambda x: m.apply("J", x), (4, g.N), free)[free]     # without the fault tangent
    place = torch.full((4 * g.N,), -1, device=DEV)
    place[free] = torch.arange(int(free.sum()), device=DEV)
    s = 1.0 / J0.diagonal().abs().sqrt()
    dK, dA = m.diagonals()
    for _ in range(case["steps"]):
        du, dp, before = torch.zeros_like(un), torch.zeros_like(pn), None
        first = None
        for it in range(60):
            law = m.law(un + du, dlie)
            b = m.residual(un, pn, du, dp, law["T"])
            size = ((b[:3] ** 2 / dK).sum() + (b[3] ** 2 / dA).sum()).sqrt().item()
            first = size if first is None else first
            if before is not None and bool((before == law["flags"]).all()) and size <= 2e-14 * first:
                break
            if before is not None and it > 30 and size <= 1e-12 * first:
                break
            before = law["flags"]
            J = J0.clone()
            pid = torch.arange(g.nb, device=DEV)
            for a in range(3):
                for c in range(3):
                    d = m.area * m.D[:, a, c]
                    for la, sa in ((g.kf, -1.0), (g.kf + 1, 1.0)):
                        for lc, sc in ((g.kf, -1.0), (g.kf + 1, 1.0)):
                            r_, c_ = place[a * g.N + la * g.nb + pid], place[c * g.N + lc * g.nb + pid]
                            ok = (r_ >= 0) & (c_ >= 0)
                            J.index_put_((r_[ok], c_[ok]), (sa * sc * d)[ok], accumulate=True)
            x = torch.zeros(4 * g.N, device=DEV, dtype=F64)
            x[free] = s * torch.linalg.solve(s[:, None] * J * s[None], s * b.reshape(-1)[free])
            du += x[:3 * g.N].view(3, g.N)
            dp += x[3 * g.N:]
        un, pn, dlie = un + du, pn + dp, law["dlie"].T.contiguous()
    host = lambda t: t.cpu().numpy()
    return dict(u=host(un), p=host(m.expand(pn)), slip=host(law["gs"]), dlie=host(law["dlie"]), flags=host(law["flags"]))


class _ExactTet:
    def __init__(self, m):
        self.m = m
        X = torch.as_tensor(m.nodes, device=DEV)
        self.t = torch.as_tensor(m.tets, device=DEV)
        e = X[self.t]
        J = (e[:, 1:] - e[:, :1])                          # rows: edge vectors
        self.V = torch.linalg.det(J).abs() / 6.0
        g = torch.linalg.inv(J)                            # columns: gradients of vertices 1..3
        G = torch.cat([-g.sum(2, keepdim=True), g], 2).transpose(1, 2)
        B = _strain(G)
        self.G, self.B, self.D = G, B, _hooke(m.E, m.nu).to(DEV)

    def matrices(self, dt):
        """Per element: K (12, 12) with columns 3 b + c, A (12, 4), S + dt C (4, 4)."""
        V, m = self.V, self.m
        K = torch.einsum("e,eia,ij,ejb->eab", V, self.B, self.D, self.B)
        A = (m.alpha * 0.25 * V)[:, None, None] * self.G.reshape(-1, 12, 1).expand(-1, 12, 4)
        S = (V / (20.0 * m.M))[:, None, None] * (1.0 + torch.eye(4, device=DEV, dtype=F64))
        C = (V * m.k / m.mu_f)[:, None, None] * torch.einsum("ead,ebd->eab", self.G, self.G)
        return K, A, S, C

    def apply(self, op, x, dt):
        N = self.m.N
        K, A, S, C = self.matrices(dt)
        u = x[:3] if op in ("KB", "AUP", "J") else None
        p = x[3] if op == "J" else x if op in ("APU", "A22") else None
        ue = None if u is None else u[:, self.t].permute(1, 2, 0).reshape(-1, 12, 1)
        pe = None if p is None else p[self.t][:, :, None]
        yu = {"KB": lambda: K @ ue, "APU": lambda: A @ pe, "J": lambda: K @ ue - A @ pe}.get(op)
        yp = {"AUP": lambda: A.transpose(1, 2) @ ue, "A22": lambda: (S + dt * C) @ pe,
              "J": lambda: A.transpose(1, 2) @ ue + (S + dt * C) @ pe}.get(op)
        out = []
        if yu is not None:
            ye = yu().reshape(-1, 4, 3)
            out += [torch.zeros(N, device=DEV, dtype=F64).index_add_(0, self.t.reshape(-1), ye[:, :, c].reshape(-1))
                    for c in range(3)]
        if yp is not None:
            out.append(torch.zeros(N, device=DEV, dtype=F64).index_add_(0, self.t.reshape(-1), yp().reshape(-1)))
        return out[0] if len(out) == 1 else torch.stack(out)

    def step(self, dt):
        """The monolithic system of one backward-Euler step from rest, solved directly."""
        m, N, t = self.m, self.m.N, self.t
        K, A, S, C = self.matrices(dt)
        J = torch.zeros((4 * N, 4 * N), device=DEV, dtype=F64)
        ud = (t[:, :, None] + N * torch.arange(3, device=DEV)).reshape(-1, 12)
        pd = t + 3 * N

        def put(rows, cols, v):
            J.index_put_((rows[:, :, None].expand_as(v), cols[:, None, :].expand_as(v)), v, accumulate=True)

        put(ud, ud, K)
        put(ud, pd, -A)
        put(pd, ud, A.transpose(1, 2))
        put(pd, pd, S + dt * C)
        f = torch.zeros(4 * N, device=DEV, dtype=F64)
        tri = torch.as_tensor(m.load_tris, device=DEV)
        X = torch.as_tensor(m.nodes, device=DEV)[tri]
        force = -m.sigma0 / 6.0 * torch.linalg.cross(X[:, 1] - X[:, 0], X[:, 2] - X[:, 0])
        for c in range(3):
            f.index_add_(0, (tri + c * N).reshape(-1), force[:, c, None].expand(-1, 3).reshape(-1))
        free = torch.as_tensor(1 - m.fixed, device=DEV).reshape(-1) > 0
        J = J[free][:, free]
        s = 1.0 / J.diagonal().abs().sqrt()
        b = s * f[free]
        J *= s[:, None]
        J *= s[None]
        LU, piv = torch.linalg.lu_factor(J)
        y = torch.linalg.lu_solve(LU, piv, b[:, None])
        for _ in range(2):
            y += torch.linalg.lu_solve(LU, piv, b[:, None] - J @ y)
        x = torch.zeros(4 * N, device=DEV, dtype=F64)
        x[free] = s * y[:, 0]
        return dict(u=x[:3 * N].view(3, N), p=x[3 * N:])


def exact(case, seed):
    kind = case["kind"]
    if kind == "tet_products":
        m = _ball(case, seed)
        e = _ExactTet(m)
        return {op: e.apply(op, _operand(op, m.u, m.p, case["dtype"]).double(), m.dt) for op in case["ops"].split(",")}
    if kind == "tet_step":
        m = _ball(case, seed)
        return _ExactTet(m).step(m.dt)
    if kind == "run" and case["nx"] * case["ny"] * case["nz"] > 600:
        return None                                        # a Newton run by other means takes minutes
    if kind == "gradient":
        return None                                        # needs the converged step, as above
    g = _grid(case, seed)
    if kind == "run":
        return _exact_run(case, g)
    u, p = _fields(g, seed)
    m = _Exact(g, 2.0)
    if kind == "residual":
        law = m.law(u)
        b = m.residual(torch.zeros_like(u), torch.zeros_like(p), u, p, law["T"])
        dK, dA = m.diagonals()
        free = m.free > 0
        rhat = (torch.where(free[:3], b[:3] ** 2 / dK, 0.0).sum() + torch.where(free[3], b[3] ** 2 / dA, 0.0).sum()).sqrt()
        law.pop("gs")
        law["flags"] = None                                # whole numbers are compared with the start's
        return dict(law=law, b=b, rhat=rhat.item())
    m.law(u)
    if kind == "products":
        return {op: m.apply(op, _operand(op, u, p, case["dtype"]).double()) for op in case["ops"].split(",")}
    free = torch.as_tensor(1 - g.fixed, device=DEV, dtype=F64)
    dK, dA = m.diagonals()
    if case["which"] == "KT":
        kd = m.area * torch.diagonal(m.D, dim1=1, dim2=2).T
        dK[:, m.up] += kd
        dK[:, m.lo] += kd
        return _cg(lambda x: m.apply("KT", x), 1e5 * u * free[:3], m.free[:3] / dK, 1e-13, 8000)
    b = 1e-15 * p * free[3] * m.free[3]
    return _cg(lambda x: m.apply("A22", x), b, torch.where(m.free[3] > 0, 1.0 / dA, 0.0), 1e-14, 8000)
