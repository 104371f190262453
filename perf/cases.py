"""What is timed: the work that a user of the solver library has it do, each
case one pass through the public entry points of the Python binding.

Kinds of cases
  solve     one load step from rest, ``Mesh.solve`` (Cook's membrane, the
            displacement form; NK, iNK, B or iB; FP64 or mixed FP32)
  twist     the same for the Taylor-Hood u-p form of the twist test
  newmark   one time step of the elastodynamic heartbeat
  batch     many small solves in one ``batch_solve``
  residual  ``Mesh.residual``: the nonlinear residual at a deformed state
  operator  ``Mesh.tangent`` (with the AMG hierarchy where asked for), then
            one product with it and one application of its preconditioner:
            what every Newton iteration pays before its Krylov iterations
  spmv      ``Mesh.spmv`` with the assembled tangent
  pc        ``Mesh.pc``: one preconditioner application
  gmres     ``Mesh.gmres``: a fixed number of Krylov iterations

The mixed forms run their tangent, products and preconditioner in FP32 and
widen the result to the FP64 vector of the interface; the cases of single
products return it in FP32, the type it was computed in (narrowing back is
exact).  Solutions are FP64 whatever the form, and are solved to 1e-10 so
that they are the solution of the problem and not of a stopping rule.

``exact`` restates the discretisation in torch FP64: P1/P2 shape functions,
the potentials by automatic differentiation, block-Jacobi, restarted GMRES
and, for the small solves, Newton with a dense factorisation.
"""
import functools
import math

import numpy as np
import torch

import paper_2203_05610_gb300 as fe
import workloads as W

EDGES = ((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # The smallest call in earnest: the 729-unknown Cook membrane, one
        # load step with the method's defaults.  Latency and launches.
        dict(name="cook_p1_nk_defaults", kind="solve", order=1, nx=8, ny=8, nz=2, method="NK", precision="fp64",
             pc="bj", orthog=0, restart=500),
        # The headline workload: 848,691 unknowns, inexact BFGS, mixed FP32
        # with the AMG V-cycle (one tangent, many Krylov iterations).
        dict(name="cook_p2_ib_large", kind="solve", order=2, nx=64, ny=64, nz=8, method="iB", precision="mixed_fp32",
             pc="amg", orthog=2, restart=50),
        # The same problem family at a tenth of the size by inexact Newton:
        # a new tangent and a new AMG hierarchy in every iteration.
        dict(name="cook_p2_ink_mid", kind="solve", order=2, nx=30, ny=26, nz=6, method="iNK", precision="mixed_fp32",
             pc="amg", orthog=2, restart=50),
        # The incompressible twist, Taylor-Hood u-p: the saddle-point
        # operator, AMG inside the lower Schur preconditioner.
        dict(name="twist_up_ink", kind="twist", n=12, precision="mixed_fp32", pc="amg", orthog=2, restart=50),
        # One step of the elastodynamic heartbeat on the 149,760-tet shell
        # (P1, Guccione, follower pressure, dashpots, inertia).
        dict(name="heart_newmark_step", kind="newmark", nr=4, nc=80, nl=78, method="iNK", precision="mixed_fp32",
             pc="amg", orthog=2, restart=50),
        # Many small requests at once: one launch, one block per request.
        dict(name="batch_small", kind="batch", count=96, low=4, high=8, precision="mixed_fp32"),
        # The nonlinear residual, the only assembly of a BFGS iteration: P2
        # neo-Hookean at the headline's size, and the P1 cardiac shell.
        dict(name="residual_p2_large", kind="residual", family="cook", order=2, nx=64, ny=64, nz=8),
        dict(name="residual_heart", kind="residual", family="heart", order=1, nx=4, ny=80, nz=78),
        # What a Newton iteration pays before its Krylov iterations, in the
        # mixed form with AMG (odd sizes) and in plain FP64 with block-Jacobi.
        dict(name="operator_p2_amg_mixed", kind="operator", family="cook", order=2, nx=45, ny=41, nz=7,
             precision="mixed_fp32", pc="amg"),
        dict(name="operator_heart_fp64", kind="operator", family="heart", order=1, nx=4, ny=80, nz=78,
             precision="fp64", pc="bj"),
        # One V-cycle at the profiled size: most of an AMG solve's time.
        dict(name="pc_amg_mixed", kind="pc", family="cook", order=2, nx=48, ny=48, nz=8, precision="mixed_fp32",
             pc="amg"),
        # A fixed budget of plain FP64 GMRES iterations (the library's
        # default precision, preconditioner and orthogonalisation).
        dict(name="gmres_fp64_bj", kind="gmres", family="cook", order=2, nx=40, ny=33, nz=5, precision="fp64",
             pc="bj", orthog=0, restart=50, iters=60),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(rng, family, order, lo, hi):
    """A mesh of about exp(U(log lo, log hi)) elements with sides of its own."""
    ne = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if family == "heart":  # thin shells: circumference and length alike
        nr = rng.randint(2, 4)
        side = math.sqrt(ne / (6 * nr))
        return dict(family=family, order=order, nx=nr, ny=max(8, int(side * rng.uniform(0.9, 1.1))),
                    nz=max(6, int(side * rng.uniform(0.85, 1.05))))
    flat = rng.uniform(3.0, 8.0)  # Cook's membrane: thin in z
    side = (flat * ne / 6) ** (1 / 3)
    return dict(family=family, order=order, nx=max(4, int(side * rng.uniform(0.85, 1.15))),
                ny=max(4, int(side * rng.uniform(0.85, 1.15))), nz=max(1, int(side / flat)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "twist", "newmark", "batch", "residual", "residual", "operator", "operator",
                       "spmv", "spmv", "pc", "pc", "gmres"])
    mixed = rng.choice(["fp64", "mixed_fp32", "mixed_fp32"])
    if kind == "solve":
        small = rng.random() < 0.25  # block-Jacobi is for small problems
        s = _sizes(rng, "cook", 1, 300, 700) if small else _sizes(rng, "cook", rng.choice([1, 2, 2]), 1000, 40000)
        method = rng.choice(["NK", "iNK", "iB"] if small else ["NK", "iNK", "B", "iB"])
        return dict(kind=kind, order=s["order"], nx=s["nx"], ny=s["ny"], nz=s["nz"], method=method, precision=mixed,
                    pc="bj" if small else "amg", orthog=rng.choice([0, 2]),
                    restart=500 if small else rng.choice([50, 100]))
    if kind == "twist":
        return dict(kind=kind, n=rng.randint(4, 14), precision=mixed, pc="amg", orthog=rng.choice([0, 2]), restart=50)
    if kind == "newmark":
        s = _sizes(rng, "heart", 1, 3000, 150000)
        return dict(kind=kind, nr=s["nx"], nc=s["ny"], nl=s["nz"], method=rng.choice(["NK", "iNK", "iB"]),
                    precision=mixed, pc="amg", orthog=2, restart=50)
    if kind == "batch":
        low = rng.randint(3, 4)
        return dict(kind=kind, count=_log_int(rng, 8, 160), low=low, high=low + rng.randint(1, 2), precision=mixed)
    family, order = rng.choice([("cook", 1), ("cook", 2), ("cook", 2), ("heart", 1)])
    top = 150000 if order == 2 else 300000
    if kind == "residual":
        return dict(kind=kind, **_sizes(rng, family, order, 1000, top))
    if kind == "gmres":
        return dict(kind=kind, **_sizes(rng, family, order, 1000, top / 4), precision="fp64", pc="bj",
                    orthog=rng.choice([0, 2]), restart=rng.choice([30, 50, 100]), iters=rng.randint(20, 80))
    pc = "bj" if kind == "spmv" else rng.choice(["bj", "amg"] if kind == "operator" else ["bj", "amg", "amg"])
    return dict(kind=kind, **_sizes(rng, family, order, 2000, top / 2), precision=mixed, pc=pc)


# ---------------------------------------------------------------- geometry
@functools.lru_cache(maxsize=6)
def _workload(family, order, nx, ny, nz):
    """The geometry and loads of a mesh (plain arrays; they carry no seed)."""
    if family == "cook":
        return W.cook(nx, ny, nz, order=order, nu=0.3)
    if family == "twist":
        return W.twist(nx)
    return W.heart(nr=nx, nc=ny, nl=nz, order=order, dynamics=family == "beat", follower=family == "beat")


def _of(case):
    k = case["kind"]
    if k == "solve":
        return "cook", case["order"], case["nx"], case["ny"], case["nz"]
    if k == "twist":
        return "twist", 2, case["n"], 0, 0
    if k == "newmark":
        return "beat", 1, case["nr"], case["nc"], case["nl"]
    return case["family"], case["order"], case["nx"], case["ny"], case["nz"]


@functools.lru_cache(maxsize=6)
def _space(family, order, nx, ny, nz):
    """Nodes of the displacement space: connectivity, positions, clamped nodes."""
    w = _workload(family, order, nx, ny, nz)
    tets, x = w["tets"].astype(np.int64), w["coords"]
    group = w["dir_group"]
    nv = x.shape[0]
    if order == 1:
        return tets, x, group, None
    e = np.sort(np.stack([tets[:, list(p)] for p in EDGES], axis=1), axis=2)
    keys, inv = np.unique((e[..., 0] * nv + e[..., 1]).reshape(-1), return_inverse=True)
    a, b = keys // nv, keys % nv
    conn = np.concatenate([tets, nv + inv.reshape(-1, 6)], axis=1)
    return (conn, np.concatenate([x, 0.5 * (x[a] + x[b])]),
            np.concatenate([group, np.where(group[a] == group[b], group[a], 0)]), keys)


def _state(case, seed, x, clamped):
    """A smooth displacement with gradients of a few per cent that fades to
    zero at the clamped face (x = 0, where there is one)."""
    rng = np.random.default_rng([seed, 1])
    size = float(np.max(x.max(0) - x.min(0)))
    d = np.zeros_like(x)
    for _ in range(3):
        k = rng.uniform(-1, 1, 3) * 4.0 / size
        d += np.sin(x @ k + rng.uniform(0, 2 * math.pi))[:, None] * rng.uniform(-1, 1, 3) * size * 0.01
    if clamped.any():
        d *= x[:, :1] / size
    return d.reshape(-1)


def _load(case, seed):
    u = float(np.random.default_rng([seed, 2]).uniform())
    if case["kind"] == "twist":
        return 0.05 + 0.05 * u, 0.0
    if case["kind"] == "newmark":
        return 0.02 + 0.04 * u, 0.004 + 0.008 * u
    if case["kind"] == "solve":
        return 0.1 + 0.1 * u, 0.0
    return (0.3 + 0.4 * u, 0.02 + 0.1 * u) if case["family"] == "heart" else (0.1 + 0.1 * u, 0.0)


def _batch(case, seed):
    """The requests of a batch: small Cook membranes and cardiac shells, the
    sizes in turn, each with a load of its own."""
    rng = np.random.default_rng([seed, 3])
    out = []
    for i in range(case["count"]):
        n = case["low"] + i % (case["high"] - case["low"] + 1)
        if i % 3 < 2:
            out.append((("cook", 1, n, n, 2), (0.1 + 0.1 * rng.uniform(), 0.0), "iNK"))
        else:
            out.append((("heart", 1, 2, 2 * n, n + 2), (0.02 + 0.04 * rng.uniform(), 0.002 + 0.004 * rng.uniform()),
                        "iNK"))
    return out


# ---------------------------------------------------------------- one pass
def _options(case):
    # no absolute Krylov tolerance: 1e-10 of the first residual lies below the default one
    return dict(precision=case["precision"], pc_type=case["pc"], orthog=case["orthog"], ksp_restart=case["restart"],
                ksp_atol=0.0)


def prepare(case, seed):
    if case["kind"] == "batch":
        meshes, methods = [], []
        for geom, load, method in _batch(case, seed):
            m = fe.Mesh(_workload(*geom))
            m.set_load(*load)
            meshes.append(m)
            methods.append(method)
        opts = dict(precision=case["precision"], ksp_restart=50, ksp_atol=0.0)
        return dict(case=case, meshes=meshes, methods=methods, opts=opts)
    geom = _of(case)
    m = fe.Mesh(_workload(*geom))
    m.set_load(*_load(case, seed))
    s = dict(case=case, m=m)
    if case["kind"] in ("solve", "twist"):
        return s
    _, x, group, _ = _space(*geom)
    d = torch.from_numpy(_state(case, seed, x, group > 0)).to(m.device)
    if case["kind"] == "newmark":
        w = _workload(*geom)
        m.set_dynamics(w["rho"], w["dt"])
        s["d"], s["v"] = 0.02 * d, 0.5 * d
        s["a"] = torch.zeros_like(d)
        return s
    s["d"] = d
    if case["kind"] == "residual":
        return s
    rng = np.random.default_rng([seed, 4])
    s["x"] = torch.from_numpy(rng.standard_normal(m.ndof)).to(m.device)
    if case["pc"] != "bj":
        m.set_pc(case["pc"])
    if case["kind"] != "operator":
        m.tangent(d, case["precision"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        ds = [m.zeros() for m in s["meshes"]]
        fe.batch_solve(s["meshes"], s["methods"], ds, [1e-10] * len(ds), opts=s["opts"])
        return torch.cat(ds)
    m = s["m"]
    if kind in ("solve", "twist"):
        d, _ = m.solve("iNK" if kind == "twist" else case["method"], m.zeros(), tol=1e-10, opts=_options(case))
        return d
    if kind == "newmark":
        m.dynamics_set(s["d"], s["v"], s["a"])
        d, _ = m.solve(case["method"], s["d"].clone(), tol=1e-10, opts=_options(case))
        m.dynamics_advance(d)
        v, a = m.dynamics_get()
        return d, v, a
    if kind == "residual":
        r, norm = m.residual(s["d"])
        return r, norm
    own = (lambda t: t) if case["precision"] == "fp64" else (lambda t: t.float())
    if kind == "operator":
        m.tangent(s["d"], case["precision"])
        return own(m.spmv(s["x"])), own(m.pc(s["x"]))
    if kind == "spmv":
        return own(m.spmv(s["x"]))
    if kind == "pc":
        return own(m.pc(s["x"]))
    x, _, _ = m.gmres(s["x"], rtol=0.0, atol=0.0, restart=case["restart"], max_it=case["iters"], orthog=case["orthog"])
    return x


# ---------------------------------------------------------------- what a pass cannot do without
def _counts(family, order, nx, ny, nz):
    """Elements, nodes, 3x3 blocks (the limits of a structured Kuhn mesh)."""
    if family == "twist":
        ny = nz = nx
    hexes = nx * ny * nz
    ne = 6 * hexes
    ring = 0 if family in ("heart", "beat") else 1
    nv = (nx + 1) * (ny + ring) * (nz + 1)
    if order == 1:
        return ne, nv, 15 * nv
    return ne, nv + 7 * hexes + 3 * (nx * ny + ny * nz + nx * nz), int(27.5 * 8 * nv)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        # about 6 Newton and 120 Krylov iterations of the mean request
        n = (case["low"] + case["high"]) / 2
        nv = 3 * (n + 1) ** 2
        return dict(bytes=case["count"] * nv * 15 * 40.0 * 120, flops=case["count"] * (nv * 15 * 18.0 * 120))
    family, order, nx, ny, nz = _of(case)
    ne, nn, nb = _counts(family, order, nx, ny, nz)
    nen = 4 if order == 1 else 10
    nq = 1 if order == 1 else 4
    n = 3 * nn
    mesh = ne * (4.0 * nen + 80.0)  # connectivity and geometry of every element
    res = dict(bytes=mesh + 16.0 * n, flops=ne * nq * 400.0)
    sv = 8.0 if case.get("precision") == "fp64" else 4.0
    block = 9 * sv + 4
    if kind == "residual":
        return res
    if kind == "spmv":
        return dict(bytes=nb * block + 16.0 * n, flops=18.0 * nb)
    amg = case["pc"] != "bj"
    # a V-cycle: four passes over the fine operator, both transfers
    pc = dict(bytes=4 * nb * block + 14.0 * nn * 18 * sv + 16.0 * n, flops=4 * 18.0 * nb + 14.0 * nn * 36) if amg \
        else dict(bytes=nn * 9 * sv + 16.0 * n, flops=18.0 * nn)
    if kind == "pc":
        return pc
    tangent = dict(bytes=mesh + 8.0 * n + nb * 9 * sv, flops=ne * nq * (nen * nen * 30.0 + 1000.0))
    if amg:  # fifteen power steps, the smoothed prolongator and the Galerkin product
        tangent = dict(bytes=tangent["bytes"] + 18 * nb * block, flops=tangent["flops"] + 18.0 * nb * 15 + 300.0 * nb)
    if kind == "operator":
        return {k: tangent[k] + pc[k] + (nb * block + 16.0 * n if k == "bytes" else 18.0 * nb) for k in pc}
    # an iteration: preconditioner, product, orthogonalisation against half a restart of vectors
    if kind == "gmres":
        its, newtons, tangents, basis = case["iters"], 0, 0, min(case["iters"], case["restart"]) / 2
    else:
        method = case.get("method", "iNK")
        newtons = {"NK": 5, "iNK": 8, "B": 80, "iB": 35}[method]
        tangents = newtons if method in ("NK", "iNK") else 1
        its = {"NK": 30, "iNK": 15, "B": 0, "iB": 15}[method] * newtons * (1 if amg else 8)
        basis = 8.0 if amg else 60.0
        if method == "B":
            newtons, its = 80, 80
    it = dict(bytes=pc["bytes"] + nb * block + 8.0 * n * basis, flops=pc["flops"] + 18.0 * nb + 4.0 * n * basis)
    return {k: its * it[k] + newtons * res[k] + tangents * tangent[k] for k in res}


# ---------------------------------------------------------------- 64-bit values
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Exact:
    """The discretisation of one mesh in torch FP64."""

    def __init__(self, geom, load, time):
        w = _workload(*geom)
        conn, x, group, keys = _space(*geom)
        dev = _dev()
        self.dev, self.mat, self.time = dev, w["material"], time
        self.order = geom[1]
        self.conn = torch.from_numpy(conn).to(dev)
        self.nn = x.shape[0]
        tets = w["tets"].astype(np.int64)
        J = np.stack([w["coords"][tets[:, k]] - w["coords"][tets[:, 0]] for k in (1, 2, 3)], axis=2)
        inv = np.linalg.inv(J)
        G = np.concatenate([-inv.sum(1, keepdims=True), inv], axis=1)  # barycentric gradients
        G = torch.from_numpy(G).to(dev)
        vol = torch.from_numpy(np.linalg.det(J) / 6.0).to(dev)
        if self.order == 1:
            g = G[:, None]
        else:
            a, b = 0.5854101966249685, 0.1381966011250105
            lam = torch.full((4, 4), b, dtype=torch.float64, device=dev)
            lam.fill_diagonal_(a)
            gv = (4 * lam[None, :, :, None] - 1) * G[:, None]
            ge = [4 * (lam[None, :, p, None] * G[:, None, q] + lam[None, :, q, None] * G[:, None, p]) for p, q in EDGES]
            g = torch.cat([gv, torch.stack(ge, 2)], 2)
        self.g = g  # [elements, points, nodes, 3]
        self.nq = g.shape[1]
        self.wq = (vol / self.nq)[:, None]
        self.fib = None if w["fibers"] is None else torch.from_numpy(w["fibers"]).to(dev).view(-1, 1, 9).expand(
            -1, self.nq, 9)
        fixed = torch.zeros(self.nn, 3, dtype=torch.bool)
        for k, grp in enumerate(w["groups"]):
            for c in range(3):
                if (grp["mask"] >> c) & 1:
                    fixed[torch.from_numpy(group == k + 1), c] = True
        self.fixed = fixed.to(dev)
        self._faces(w, keys, load)

    def _faces(self, w, keys, load):
        """Dead loads and springs: the triangle's mass matrix and load vector."""
        f = w["faces"].astype(np.int64)
        nv = w["coords"].shape[0]
        x = w["coords"][f]
        n = np.cross(x[:, 1] - x[:, 0], x[:, 2] - x[:, 0])
        area2 = np.linalg.norm(n, axis=1, keepdims=True)
        N, A = n / area2, 0.5 * area2[:, 0]
        if self.order == 1:
            nodes, share = f, np.full(3, 1 / 3)
            mass = (np.ones((3, 3)) + np.eye(3)) / 12
        else:
            e = np.sort(np.stack([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]], 1), axis=2)
            nodes = np.concatenate([f, nv + np.searchsorted(keys, e[..., 0] * nv + e[..., 1])], 1)
            share = np.array([0, 0, 0, 1 / 3, 1 / 3, 1 / 3])
            mass = np.zeros((6, 6))
            mass[:3, :3] = 7 * np.eye(3) - 1
            mass[3:, 3:] = 16 + 16 * np.eye(3)
            for v in range(3):
                mass[v, 3 + (v + 1) % 3] = mass[3 + (v + 1) % 3, v] = -4
            mass /= 180
        kind, data = w["face_kind"], w["face_data"]
        t = np.where((kind == W.FACE_TRACTION)[:, None], data, 0) - np.where((kind == W.FACE_PRESSURE)[:, None],
                                                                             data[:, :1] * N, 0)
        F = load * A[:, None, None] * share[None, :, None] * t[:, None]
        self.fext = torch.zeros(self.nn, 3, dtype=torch.float64, device=self.dev)
        self.fext.index_add_(0, torch.from_numpy(nodes.reshape(-1)).to(self.dev),
                             torch.from_numpy(F.reshape(-1, 3)).to(self.dev))
        rob = kind == W.FACE_ROBIN
        NN = N[:, :, None] * N[:, None]
        C = data[:, 0, None, None] * NN + data[:, 1, None, None] * (np.eye(3) - NN)
        K = (A[:, None, None, None, None] * mass[None, :, :, None, None] * C[:, None, None])[rob]
        self.snode = torch.from_numpy(nodes[rob]).to(self.dev)
        self.K = torch.from_numpy(K).to(self.dev)

    def _psi(self, F, fib):
        m = self.mat
        c = lambda i, j, k, l: F[i] * F[j] - F[k] * F[l]  # noqa: E731
        J = F[0] * c(4, 8, 5, 7) + F[1] * c(5, 6, 3, 8) + F[2] * c(3, 7, 4, 6)
        I1 = (F * F).sum()
        if m["kind"] == W.MAT_COOK_NH:
            mu = m["E"] / (2 * (1 + m["nu"]))
            kap = 2 * mu * m["nu"] / (1 - 2 * m["nu"]) + 2 * mu / 3
            return 0.5 * mu * (I1 * J ** (-2 / 3) - 3) + 0.25 * kap * (J * J - 1 - 2 * torch.log(J))
        Fm, R = F.view(3, 3), fib.view(3, 3)
        E = 0.5 * (Fm.T @ Fm - torch.eye(3, dtype=F.dtype, device=F.device))
        Ef = R @ E @ R.T
        B = torch.full((3, 3), m["bt"], dtype=F.dtype, device=F.device)
        B[0] = m["bfs"]
        B[:, 0] = m["bfs"]
        B[0, 0] = m["bf"]
        act = m["Ta_peak"] * max(math.sin(2 * math.pi * self.time / m["period"]), 0.0)
        return (0.5 * m["C"] * (torch.exp((B * Ef * Ef).sum()) - 1) + 0.5 * m["kappa"] * (J - 1) * torch.log(J)
                + act * torch.linalg.norm(Fm @ R[0]))

    def _points(self, d, what):
        """``what`` (a derivative of psi) at every quadrature point."""
        u = d.view(-1, 3)[self.conn]
        F = torch.einsum("eai,eqaj->eqij", u, self.g) + torch.eye(3, dtype=torch.float64, device=self.dev)
        F = F.reshape(-1, 9)
        fib = torch.zeros(F.shape[0], 1, dtype=F.dtype, device=self.dev) if self.fib is None \
            else self.fib.reshape(-1, 9)
        f = torch.func.vmap(what)
        return torch.cat([f(a, b) for a, b in zip(F.split(200000), fib.split(200000))])

    def _scatter(self, P):
        """sum over points of w P grad N_a, added up at the nodes."""
        e = torch.einsum("eqij,eqaj,eq->eai", P.view(-1, self.nq, 3, 3), self.g, self.wq.expand(-1, self.nq))
        out = torch.zeros(self.nn, 3, dtype=torch.float64, device=self.dev)
        return out.index_add_(0, self.conn.reshape(-1), e.reshape(-1, 3))

    def _springs(self, x):
        y = torch.zeros_like(x)
        if len(self.snode):
            e = torch.einsum("fabij,fbj->fai", self.K, x[self.snode])
            y.index_add_(0, self.snode.reshape(-1), e.reshape(-1, 3))
        return y

    def residual(self, d):
        r = self._scatter(self._points(d, torch.func.grad(self._psi))) - self.fext + self._springs(d.view(-1, 3))
        return torch.where(self.fixed, 0.0, r).reshape(-1)

    def tangent(self, d):
        self.A = self._points(d, torch.func.hessian(self._psi)).view(-1, self.nq, 3, 3, 3, 3)
        D = torch.zeros(self.nn, 3, 3, dtype=torch.float64, device=self.dev)
        e = torch.einsum("eqijkl,eqaj,eqal,eq->eaik", self.A, self.g, self.g, self.wq.expand(-1, self.nq))
        D.index_add_(0, self.conn.reshape(-1), e.reshape(-1, 3, 3))
        if len(self.snode):
            i = torch.arange(self.snode.shape[1], device=self.dev)
            D.index_add_(0, self.snode.reshape(-1), self.K[:, i, i].reshape(-1, 3, 3))
        free = (~self.fixed).double()
        D = D * free[:, :, None] * free[:, None] + torch.diag_embed(1 - free)
        self.D = torch.linalg.inv(D)

    def spmv(self, x):
        x = x.view(-1, 3)
        z = torch.where(self.fixed, 0.0, x)
        dF = torch.einsum("eai,eqaj->eqij", z[self.conn], self.g)
        y = self._scatter(torch.einsum("eqijkl,eqkl->eqij", self.A, dF)) + self._springs(z)
        return torch.where(self.fixed, x, y).reshape(-1)

    def pc(self, x):
        return torch.einsum("aij,aj->ai", self.D, x.view(-1, 3)).reshape(-1)

    def gmres(self, b, restart, iters):
        """Right-preconditioned GMRES(restart), ``iters`` iterations from zero."""
        x = torch.zeros_like(b)
        done = 0
        while done < iters:
            r = b - self.spmv(x)
            beta = r.norm()
            k = min(restart, iters - done)
            V, H = [r / beta], torch.zeros(k + 1, k, dtype=torch.float64)
            for j in range(k):
                w = self.spmv(self.pc(V[j]))
                for _ in range(2):
                    for i in range(j + 1):
                        h = torch.dot(w, V[i])
                        H[i, j] += float(h)
                        w = w - h * V[i]
                H[j + 1, j] = float(w.norm())
                V.append(w / w.norm())
            rhs = torch.zeros(k + 1, dtype=torch.float64)
            rhs[0] = float(beta)
            y = torch.linalg.lstsq(H, rhs[:, None]).solution[:, 0]
            x = x + self.pc(sum(float(c) * v for c, v in zip(y, V)))
            done += k
        return x

    def solution(self):
        """Newton from rest with a dense factorisation."""
        n = 3 * self.nn
        d = torch.zeros(n, dtype=torch.float64, device=self.dev)
        start = None
        free = (~self.fixed).reshape(-1)
        for _ in range(40):
            r = self.residual(d)
            start = start or float(r.norm())
            if float(r.norm()) <= 1e-13 * start:
                break
            self.tangent(d)
            e = torch.einsum("eqijkl,eqaj,eqbl,eq->eaibk", self.A, self.g, self.g, self.wq.expand(-1, self.nq))
            at = (3 * self.conn[:, :, None] + torch.arange(3, device=self.dev)).reshape(len(self.conn), -1)
            K = torch.zeros(n * n, dtype=torch.float64, device=self.dev)
            m = at.shape[1]
            K.index_add_(0, (at[:, :, None] * n + at[:, None]).reshape(-1), e.reshape(-1, m * m).reshape(-1))
            if len(self.snode):
                at = (3 * self.snode[:, :, None] + torch.arange(3, device=self.dev)).reshape(len(self.snode), -1)
                K.index_add_(0, (at[:, :, None] * n + at[:, None]).reshape(-1),
                             self.K.permute(0, 1, 3, 2, 4).reshape(-1))
            K = K.view(n, n)[free][:, free]
            d[free] -= torch.linalg.solve(K, r[free])
        return d


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        if case["count"] > 100:
            return None
        return torch.cat([_Exact(g, *load).solution() for g, load, _ in _batch(case, seed)])
    if kind in ("twist", "newmark"):
        return None
    geom = _of(case)
    _, x, group, _ = _space(*geom)
    n = 3 * x.shape[0]
    if kind == "solve":
        return _Exact(geom, *_load(case, seed)).solution() if n <= 4000 else None
    E = _Exact(geom, *_load(case, seed))
    d = torch.from_numpy(_state(case, seed, x, group > 0)).to(E.dev)
    if kind == "residual":
        r = E.residual(d)
        return r, float(r.norm())
    if kind == "pc" and case["pc"] != "bj":
        return None
    E.tangent(d)
    b = torch.from_numpy(np.random.default_rng([seed, 4]).standard_normal(n)).to(E.dev)
    if kind == "spmv":
        return E.spmv(b)
    if kind == "pc":
        return E.pc(b)
    if kind == "operator":
        return E.spmv(b), None if case["pc"] != "bj" else E.pc(b)
    return E.gmres(b, case["restart"], case["iters"])
