"""The work that users of the tangent solver have it do, as timed cases.

A user builds a ``Problem`` from a mesh, keeps it and a ``BDDC`` context for
the whole simulation, and calls, in every Newton step or inside a Krylov
loop of their own: ``newton_step`` (assembly, BDDC setup, GMRES, update),
``residual``, ``assemble_tangent``, ``spmv``, ``BDDC.setup``, ``BDDC.apply``
and ``BDDC.gmres``.  Each case is one such call (or the two that belong
together) on one mesh.  The meshes are those of the benchmark (8^3 Q1 cube,
48x48x12 Q1 slab, 24x24x6 Q2 slab, P1 and P2 left ventricles) and, for the
ventricles, the same generator at sizes whose host-side preparation stays
short; the drawn cases spread over the same families, sizes and options.

``exact`` evaluates the same residuals, tangent products and Newton updates
from the strain energy in plain torch FP64 (automatic differentiation, block
tridiagonal elimination); it uses nothing but the mesh arrays.
"""
import functools
import math

import numpy as np
import torch

import paper_2208_06191_gb300 as pkg
import workloads

F64 = torch.float64


# ------------------------------------------------------------------- cases

def _slab(name, kind, order, n, parts, precision, primal, **kw):
    return dict(name=name, kind=kind, mesh="slab", order=order, nx=n[0], ny=n[1], nz=n[2],
                px=parts[0], py=parts[1], pz=parts[2], precision=precision, primal=primal,
                **{**dict(levels=2, scaling="counting", coarse="galerkin", restart=100, timed=False,
                          jitter=0.0), **kw})


def _lv(name, kind, order, n, n_parts, precision, primal, **kw):
    return dict(name=name, kind=kind, mesh="lv", order=order, nt=n[0], ntheta=n[1], nu=n[2],
                n_parts=n_parts, precision=precision, primal=primal,
                **{**dict(levels=2, n_parts2=0, n_layers=1, scaling="counting", coarse="galerkin",
                          restart=1000, timed=False), **kw})


def listed():
    return [
        # one Newton step of the smallest workload: launches and latency count
        _slab("newton_cube8_q1_f64", "newton", 1, (8, 8, 8), (2, 2, 2), "f64", "V"),
        # the Newton step of the two slab workloads, FP32 local operators
        # (the benchmark's setting) and FP64 ones (the library's default)
        _slab("newton_slab48_q1_f32", "newton", 1, (48, 48, 12), (4, 4, 4), "f32", "VE"),
        _slab("newton_slab48_q1_f64", "newton", 1, (48, 48, 12), (4, 4, 4), "f64", "VE"),
        _slab("newton_slab24_q2_f32", "newton", 2, (24, 24, 6), (8, 4, 2), "f32", "VEF"),
        # the Newton step on the reduced P1 ventricle, uneven subdomains,
        # two-level
        _lv("newton_lv_p1_f64", "newton", 1, (5, 64, 32), 64, "f64", "VEF"),
        # ... and on a P2 ventricle, three-level with FP32 local operators:
        # the benchmark's configuration on a mesh a fifth as large
        _lv("newton_lv_p2_ml_f32", "newton", 2, (5, 80, 72), 512, "f32", "VEF", levels=3,
            n_parts2=16, n_layers=2),
        # a solve with another right-hand side on a set-up preconditioner
        # (deluxe scaling, the robust choice on the ventricle)
        _lv("gmres_lv_p1_dlx_f32", "gmres", 1, (5, 64, 32), 64, "f32", "VEF", scaling="deluxe"),
        # refreshing the preconditioner for a new tangent and applying it
        # once, ragged mesh and boxes, separate left and right coarse bases
        _slab("precond_ragged_q1_petrov_f64", "precond", 1, (23, 19, 9), (4, 3, 2), "f64", "VEF",
              coarse="petrov", jitter=0.15),
        # one application inside a Krylov loop of the user's own
        _lv("apply_lv_p2_ml_f64", "apply", 2, (5, 64, 32), 128, "f64", "VEF", levels=3, n_parts2=8,
            n_layers=2),
        # residual and tangent of the P2 ventricle and one product with it
        _lv("tangent_lv_p2", "tangent", 2, (5, 104, 96), 64, "f64", "VEF"),
        # residual alone (line search, time stepping): backward-Euler state
        # with inertia and Robin faces on a Q2 slab
        _slab("residual_q2_time", "residual", 2, (23, 21, 6), (2, 2, 1), "f64", "VEF", timed=True,
              jitter=0.1),
        # the operator product of a Krylov loop of the user's own, P1
        # ventricle with a tangent larger than the L2 cache
        _lv("spmv_lv_p1", "spmv", 1, (9, 160, 112), 64, "f64", "VEF"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _dense_work(c):
    """Sum over the subdomains of the cube of their unknowns, roughly: what
    the dense local operators of a setup cost."""
    o = c["order"]
    if c["mesh"] == "slab":
        ns, parts = 3.0, c["px"] * c["py"] * c["pz"]
        for n, p in ((c["nx"], c["px"]), (c["ny"], c["py"]), (c["nz"], c["pz"])):
            ns *= o * math.ceil(n / p) + 1
    else:
        parts = c["n_parts"]
        ns = 3 * 1.5 * c["ntheta"] * c["nu"] * o * o * (o * (c["nt"] - 1) + 1) / parts
    return parts * ns ** 3


def draw(rng):
    while True:
        c = _draw(rng)
        # at most half of the 48x48x12 slab's (64 boxes of 2028 unknowns)
        if c["kind"] not in ("newton", "gmres", "precond", "apply") or _dense_work(c) <= 32 * 2028.0 ** 3:
            return c


def _draw(rng):
    kind = rng.choice(["newton"] * 4 + ["gmres", "precond", "precond", "apply", "tangent", "residual",
                                        "spmv"])
    precision = rng.choice(["f32", "f64"]) if kind in ("newton", "gmres") else "f64"
    mesh = rng.choice(["slab", "lv"])
    order = rng.choice([1, 1, 2])
    scaling = rng.choice(["counting", "counting", "deluxe"])
    coarse = rng.choice(["galerkin", "galerkin", "petrov"])
    local = kind in ("newton", "gmres", "precond", "apply")
    if mesh == "slab":
        # boxes of h elements per edge (Q2 elements carry eight Q1 ones)
        top = 12 if order == 1 else 6
        h = rng.randint(3, top) if order == 1 else rng.randint(2, 4)
        if local:
            px, py, pz = rng.randint(2, 5), rng.randint(2, 4), rng.randint(1, 3)
            n = (max(4, px * h - rng.randint(0, 2)), max(4, py * h - rng.randint(0, 1)), max(3, pz * min(h, 5)))
        else:
            px, py, pz = 2, 2, 1
            n = (_log_int(rng, 6, 48 // order), _log_int(rng, 6, 48 // order), rng.randint(3, top))
        c = _slab("drawn", kind, order, n, (px, py, pz), precision, rng.choice(["VE", "VEF"]),
                  scaling=scaling, coarse=coarse, jitter=rng.choice([0.0, 0.1, 0.15]),
                  timed=kind == "residual" and rng.random() < 0.5)
    else:
        nu = _log_int(rng, 16, 40 if local else 96 // order)
        ntheta = 8 * rng.randint(max(2, nu // 8), max(3, nu // 4))
        nt = rng.choice([3, 5])
        surf = ntheta * nu * order * order
        if not local:
            n_parts, levels, n2, layers = 8, 2, 0, 1
        else:
            per = rng.randint(24, 60) * (4 if order == 1 else 3)  # surface nodes per patch
            levels = rng.choice([2, 3])
            n2 = rng.choice([4, 8]) if levels == 3 else 0
            patches = max(8, int(surf / per)) // max(n2, 1) * max(n2, 1)
            layers = rng.choice([1, 2]) if order == 2 else 1
            n_parts = max(patches, 8) * layers
            if levels == 3:
                scaling = "counting"
        c = _lv("drawn", kind, order, (nt, ntheta, nu), n_parts, precision, "VEF", levels=levels,
                n_parts2=n2, n_layers=layers, scaling=scaling, coarse=coarse, restart=rng.choice([100, 300, 1000]))
    del c["name"]
    return c


@functools.lru_cache(maxsize=4)
def _mesh_of(items):
    c = dict(items)
    if c["mesh"] == "slab":
        h = 1.0 / 12.0 if c["order"] == 1 else 1.0 / 6.0
        prob = workloads.slab_problem(c["nx"], c["ny"], c["nz"], order=c["order"],
                                      lengths=(c["nx"] * h, c["ny"] * h, c["nz"] * h),
                                      parts=(c["px"], c["py"], c["pz"]), jitter=c["jitter"],
                                      primal=c["primal"], load_steps=4)
    else:
        prob = workloads.lv_problem(nt=c["nt"], ntheta=c["ntheta"], nu=c["nu"], order=c["order"],
                                    jitter=0.1, n_parts=c["n_parts"], n_parts2=c["n_parts2"] or None,
                                    n_layers=c["n_layers"], primal=c["primal"], load_steps=8,
                                    gamma=0.25 * 6.0e4)
    if c["timed"]:
        nx, ny, nz = c["nx"], c["ny"], c["nz"]
        side = np.arange(nx * ny * nz)
        x0 = side[side % nx == 0]
        prob["rho"] = 1000.0
        prob["robin_faces"] = np.stack([x0, 0 * x0, x0 % 2], axis=1)
        prob["robin"] = [dict(k_perp=2e5, k_par=2e4, c_perp=1e4, c_par=2e3),
                         dict(k_perp=1e5, k_par=1e4, c_perp=5e3, c_par=1e3)]
    return prob


def _mesh(case):
    return _mesh_of(tuple(sorted((k, v) for k, v in case.items() if k != "name")))


DT = 0.01


def _inputs(case, seed):
    """Displacement (free DoFs), load factor, vectors and time state, from
    the seed: a smooth field that vanishes at the clamped face, of the few
    percent of strain that a load step's Newton states have."""
    prob = _mesh(case)
    rng = np.random.default_rng(seed)
    X = np.asarray(prob["coords"])
    free = np.setdiff1d(np.arange(len(X)), prob["dirichlet_nodes"])
    Xf = X[free]
    scale = 1.0 if case["mesh"] == "slab" else 1.0 / 0.03
    n = 3 * len(free)

    def field(amp):
        k = rng.uniform(0.5, 1.5, 3)
        ph = rng.uniform(0.0, 2.0 * np.pi, 3)
        return (amp * Xf[:, 2:3] * np.sin(k * Xf * scale + ph)).reshape(-1)

    # (the thin ventricle wall takes less before its tangent loses stability)
    d = field(0.015 if case["mesh"] == "slab" else 0.002)
    load = float(rng.uniform(0.25, 0.75)) if case["mesh"] == "slab" else float(rng.uniform(0.1, 0.15))
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    x = torch.randn(n, dtype=F64, device="cuda", generator=g)
    dev = functools.partial(torch.as_tensor, dtype=F64, device="cuda")
    d_prev = d_prev2 = None
    if case["timed"]:
        step = field(0.001)
        d_prev, d_prev2 = dev(d - step), dev(d - 1.9 * step)
    return dict(prob=prob, free=free, d=dev(d), load=load, x=x, d_prev=d_prev, d_prev2=d_prev2)


def _precision(case):
    return pkg.FP32 if case["precision"] == "f32" else pkg.FP64


def _multilevel(case, prob):
    if case["levels"] < 3:
        return {}
    return dict(levels=3, part2=prob["part2"], n_parts2=prob["n_parts2"], primal2="VEF",
                precision2=_precision(case))


def prepare(case, seed):
    s = _inputs(case, seed)
    prob = s["prob"]
    P = pkg.Problem(prob)
    s.update(case=case, P=P, out=torch.empty_like(s["d"]), out2=torch.empty_like(s["d"]))
    if case["timed"]:
        P.set_time_state(DT, s["d_prev"], s["d_prev2"])
    if case["kind"] in ("newton", "gmres", "precond", "apply", "spmv"):
        r = torch.empty_like(s["d"])
        P.assemble_tangent(s["d"], s["load"], r)
        s["b"] = -r
    if case["kind"] in ("newton", "gmres", "precond", "apply"):
        common = dict(precision=_precision(case), primal=case["primal"], scaling=case["scaling"],
                      coarse=case["coarse"], **_multilevel(case, prob))
        s["pc"] = pkg.BDDC(P, **common).setup()
        if case["kind"] == "newton":
            s["options"] = pkg.SolveOptions(restart=case["restart"], max_gmres=3000, **common)
    return s


def run(s):
    case, P = s["case"], s["P"]
    kind = case["kind"]
    if kind == "newton":
        d = s["d"].clone()
        P.newton_step(d, s["load"], s["options"], s["pc"])
        return d
    if kind == "gmres":
        s["pc"].gmres(s["b"], s["out"], restart=case["restart"], max_iters=3000)
        return s["out"]
    if kind == "precond":
        s["pc"].setup()
        return s["pc"].apply(s["x"], s["out"])
    if kind == "apply":
        return s["pc"].apply(s["x"], s["out"])
    if kind == "tangent":
        P.assemble_tangent(s["d"], s["load"], s["out"])
        P.spmv(s["x"], s["out2"])
        return s["out"], s["out2"]
    if kind == "residual":
        return P.residual(s["d"], s["load"], s["out"])
    return P.spmv(s["x"], s["out"])


def work(case):
    """Bytes: the mesh arrays (coordinates, connectivity, nodal fibres) and
    the input and output vectors once, for a product with the tangent its
    blocks once (72 bytes and a column index each).  Flops: the contraction
    of the stress (and its derivative, over the symmetric half of the
    element matrix) with the shape gradients, one product with the tangent
    for each kind that needs one; a solve needs more, by an amount that
    depends on the state."""
    prob = _mesh(case)
    elems = np.asarray(prob["elems"])
    n_nodes, (n_el, n_en) = len(prob["coords"]), elems.shape
    n_qp = {"P1": 1, "P2": 4, "Q1": 8, "Q2": 27}[prob["elem_type"]]
    n = 3 * (n_nodes - len(prob["dirichlet_nodes"]))
    mesh = n_nodes * 24 + elems.size * 4 + (n_nodes * 48 if prob["fibers"]["kind"] == "nodal" else 0)
    # blocks of the tangent: ordered node pairs that share an element
    blocks = n_nodes * {"P1": 15, "P2": 29, "Q1": 27, "Q2": 64}[prob["elem_type"]]
    res_flops = n_el * n_qp * n_en * 36.0
    tan_flops = 2.0 * n_el * n_qp * (81.0 * n_en + 27.0 * n_en * (n_en + 1) / 2)
    kind = case["kind"]
    if kind == "spmv":
        return dict(bytes=blocks * 76.0 + 16.0 * n, flops=18.0 * blocks)
    if kind == "residual":
        return dict(bytes=mesh + 16.0 * n + (16.0 * n if case["timed"] else 0), flops=res_flops)
    if kind == "tangent":
        return dict(bytes=mesh + 32.0 * n + 2 * blocks * 76.0, flops=res_flops + tan_flops + 18.0 * blocks)
    if kind == "newton":
        return dict(bytes=mesh + 16.0 * n + 2 * blocks * 76.0, flops=res_flops + tan_flops + 18.0 * blocks)
    return dict(bytes=blocks * 76.0 + 16.0 * n, flops=18.0 * blocks)


# ----------------------------------------------------- the same in plain torch

def _shapes(kind):
    """(N [q, a], dN [q, a, 3], w [q]) of the volume rule."""
    if kind in ("Q1", "Q2"):
        k = int(kind[1])
        x, w = np.polynomial.legendre.leggauss(k + 1)
        nodes = np.linspace(-1.0, 1.0, k + 1)
        L = [np.poly1d(np.poly(np.delete(nodes, i))) / np.prod(nodes[i] - np.delete(nodes, i)) for i in range(k + 1)]
        V = np.array([[p(t) for p in L] for t in x])
        D = np.array([[p.deriv()(t) for p in L] for t in x])
        q = [(a, b, c) for c in range(k + 1) for b in range(k + 1) for a in range(k + 1)]
        N = np.array([[V[i[0], j[0]] * V[i[1], j[1]] * V[i[2], j[2]] for j in q] for i in q])
        dN = np.array([[[D[i[0], j[0]] * V[i[1], j[1]] * V[i[2], j[2]],
                         V[i[0], j[0]] * D[i[1], j[1]] * V[i[2], j[2]],
                         V[i[0], j[0]] * V[i[1], j[1]] * D[i[2], j[2]]] for j in q] for i in q])
        return N, dN, np.array([w[i[0]] * w[i[1]] * w[i[2]] for i in q])
    if kind == "P1":
        pts, w = [[0.25, 0.25, 0.25]], np.array([1.0 / 6.0])
    else:
        a, b = (5 + 3 * math.sqrt(5)) / 20, (5 - math.sqrt(5)) / 20
        pts, w = [[b, b, b], [a, b, b], [b, a, b], [b, b, a]], np.full(4, 1.0 / 24.0)
    G = np.array([[-1.0, -1, -1], [1, 0, 0], [0, 1, 0], [0, 0, 1]])
    edges = [(0, 1), (1, 2), (0, 2), (0, 3), (1, 3), (2, 3)]
    Ns, dNs = [], []
    for p in pts:
        L = np.array([1 - sum(p), *p])
        if kind == "P1":
            Ns.append(L)
            dNs.append(G)
        else:
            Ns.append(np.concatenate([L * (2 * L - 1), [4 * L[i] * L[j] for i, j in edges]]))
            dNs.append(np.concatenate([(4 * L - 1)[:, None] * G, [4 * (L[j] * G[i] + L[i] * G[j]) for i, j in edges]]))
    return np.array(Ns), np.array(dNs), w


def _face_shapes(kind):
    """(N, dN/ds, dN/dt [q, a], w) of the face rule and the local nodes of
    every face, ordered so that x_s x x_t points outwards."""
    if kind in ("Q1", "Q2"):
        k = int(kind[1])
        x, w = np.polynomial.legendre.leggauss(k + 1)
        nodes = np.linspace(-1.0, 1.0, k + 1)
        L = [np.poly1d(np.poly(np.delete(nodes, i))) / np.prod(nodes[i] - np.delete(nodes, i)) for i in range(k + 1)]
        V = np.array([[p(t) for p in L] for t in x])
        D = np.array([[p.deriv()(t) for p in L] for t in x])
        q = [(a, b) for b in range(k + 1) for a in range(k + 1)]
        N = np.array([[V[i[0], j[0]] * V[i[1], j[1]] for j in q] for i in q])
        S = np.array([[D[i[0], j[0]] * V[i[1], j[1]] for j in q] for i in q])
        T = np.array([[V[i[0], j[0]] * D[i[1], j[1]] for j in q] for i in q])
        m = k + 1
        faces = []
        for f in range(6):
            ax, hi = f // 2, f % 2
            e, g = (ax + 1) % 3, (ax + 2) % 3
            if not hi:
                e, g = g, e
            row = []
            for i, j in q:
                idx = [0, 0, 0]
                idx[ax], idx[e], idx[g] = k * hi, i, j
                row.append(idx[0] + m * (idx[1] + m * idx[2]))
            faces.append(row)
        return N, S, T, np.array([w[i[0]] * w[i[1]] for i in q]), faces
    corners = [(1, 2, 3), (0, 3, 2), (0, 1, 3), (0, 2, 1)]
    mid = {(0, 1): 4, (1, 2): 5, (0, 2): 6, (0, 3): 7, (1, 3): 8, (2, 3): 9}
    G = np.array([[-1.0, -1.0], [1, 0], [0, 1]])
    edges = [(0, 1), (1, 2), (0, 2)]
    if kind == "P1":
        pts, w, faces = [[1 / 3, 1 / 3]], np.array([0.5]), [list(c) for c in corners]
    else:
        pts, w = [[1 / 6, 1 / 6], [2 / 3, 1 / 6], [1 / 6, 2 / 3]], np.full(3, 1 / 6)
        faces = [list(c) + [mid[tuple(sorted((c[i], c[j])))] for i, j in edges] for c in corners]
    Ns, dNs = [], []
    for p in pts:
        L = np.array([1 - sum(p), *p])
        if kind == "P1":
            Ns.append(L)
            dNs.append(G)
        else:
            Ns.append(np.concatenate([L * (2 * L - 1), [4 * L[i] * L[j] for i, j in edges]]))
            dNs.append(np.concatenate([(4 * L - 1)[:, None] * G, [4 * (L[j] * G[i] + L[i] * G[j]) for i, j in edges]]))
    D = np.array(dNs)
    return np.array(Ns), D[:, :, 0], D[:, :, 1], w, faces


class _Plain:
    """Residual and tangent of the model from its energy, in torch FP64."""

    def __init__(self, s, case):
        prob = s["prob"]
        dev = functools.partial(torch.as_tensor, dtype=F64, device="cuda")
        self.load, self.case = s["load"], case
        self.X = dev(np.asarray(prob["coords"]))
        self.elems = torch.as_tensor(np.asarray(prob["elems"]), dtype=torch.long, device="cuda")
        N, dN, w = (dev(a) for a in _shapes(prob["elem_type"]))
        Xe = self.X[self.elems]
        J = torch.einsum("eai,qaj->eqij", Xe, dN)
        self.G = torch.einsum("qaj,eqji->eqai", dN, torch.linalg.inv(J))
        self.wd = w * torch.linalg.det(J)
        self.N = N
        fib = prob["fibers"]
        if fib["kind"] == "nodal":
            f = torch.einsum("qa,eai->eqi", N, dev(np.asarray(fib["f"]))[self.elems])
            n = torch.einsum("qa,eai->eqi", N, dev(np.asarray(fib["n"]))[self.elems])
            f = f / f.norm(dim=-1, keepdim=True)
            n = n - (n * f).sum(-1, keepdim=True) * f
            n = n / n.norm(dim=-1, keepdim=True)
            self.R = torch.stack([f, torch.linalg.cross(n, f), n], dim=-1)
        else:
            z = torch.einsum("qa,ea->eq", N, Xe[..., 2])
            al = fib["alpha0"] + (fib["alpha1"] - fib["alpha0"]) * (z - fib["z0"]) / (fib["z1"] - fib["z0"])
            c, t, o, i = torch.cos(al), torch.sin(al), torch.zeros_like(al), torch.ones_like(al)
            self.R = torch.stack([c, -t, o, t, c, o, o, o, i], dim=-1).reshape(*al.shape, 3, 3)
        m = prob["material"]
        self.W = dev([[m["bff"], m["bfs"], m["bfn"]], [m["bfs"], m["bss"], m["bsn"]], [m["bfn"], m["bsn"], m["bnn"]]])
        self.C, self.B = m["C"], m["B"]
        self.gamma, self.p = self.load * prob["gamma"], self.load * prob["pressure"]
        fN, fS, fT, fw, faces = _face_shapes(prob["elem_type"])
        self.fN, self.fS, self.fT, self.fw = dev(fN), dev(fS), dev(fT), dev(fw)
        faces = torch.as_tensor(faces, dtype=torch.long, device="cuda")

        def nodes_of(lst):
            lst = torch.as_tensor(np.asarray(lst), dtype=torch.long, device="cuda")
            return torch.gather(self.elems[lst[:, 0]], 1, faces[lst[:, 1]])

        self.pf = nodes_of(prob["pressure_faces"])
        self.free = torch.as_tensor(s["free"], device="cuda")
        self.time = None
        if case["timed"]:
            self.time = (self.full(s["d_prev"]), self.full(s["d_prev2"]))
            self.rho = prob["rho"]
            rf = np.asarray(prob["robin_faces"])
            self.rf = nodes_of(rf[:, :2])
            par = dev([[q[k] for k in ("k_perp", "k_par", "c_perp", "c_par")] for q in prob["robin"]])
            self.rp = par[torch.as_tensor(rf[:, 2], dtype=torch.long, device="cuda")]

    def full(self, d):
        u = torch.zeros_like(self.X)
        u[self.free] = d.reshape(-1, 3)
        return u

    def energy(self, ue, G, R, wd):
        """Strain and active energy of elements (any leading axes)."""
        F = torch.eye(3, dtype=F64, device="cuda") + torch.einsum("...ai,...qaj->...qij", ue, G)
        E = 0.5 * (F.transpose(-1, -2) @ F - torch.eye(3, dtype=F64, device="cuda"))
        Ep = R.transpose(-1, -2) @ E @ R
        Q = (self.W * Ep * Ep).sum((-1, -2))
        c = torch.linalg.cross(F[..., 0, :], F[..., 1, :], dim=-1)
        J = (c * F[..., 2, :]).sum(-1)
        Ff = (F @ R[..., :, :1])[..., 0]
        W = 0.5 * self.C * (torch.exp(Q) - 1) + 0.5 * self.B * (J - 1) * torch.log(J) + self.gamma * torch.sqrt((Ff * Ff).sum(-1))
        return (wd * W).sum(-1)

    def pressure(self, xf):
        """Follower-pressure residual of faces with deformed nodes xf."""
        s = torch.einsum("qa,...ai->...qi", self.fS, xf)
        t = torch.einsum("qa,...ai->...qi", self.fT, xf)
        return self.p * torch.einsum("q,qa,...qi->...ai", self.fw, self.fN, torch.linalg.cross(s, t, dim=-1))

    def potential(self, u):
        e = self.energy(u[self.elems], self.G, self.R, self.wd).sum()
        if self.time is not None:
            dp, dpp = self.time
            a = torch.einsum("qa,eai->eqi", self.N, (u - 2 * dp + dpp)[self.elems])
            e = e + 0.5 * self.rho / DT ** 2 * (self.wd * (a * a).sum(-1)).sum()
            Xf = self.X[self.rf]
            A = torch.linalg.cross(torch.einsum("qa,fai->fqi", self.fS, Xf), torch.einsum("qa,fai->fqi", self.fT, Xf), dim=-1)
            area = A.norm(dim=-1)
            n = A / area[..., None]
            uq = torch.einsum("qa,fai->fqi", self.fN, u[self.rf])
            vq = torch.einsum("qa,fai->fqi", self.fN, (u - dp)[self.rf])
            k = self.rp[:, None, :]

            def split(v):
                vn = (v * n).sum(-1)
                return vn * vn, (v * v).sum(-1) - vn * vn

            (un, ut), (vn, vt) = split(uq), split(vq)
            dens = k[..., 0] * un + k[..., 1] * ut + (k[..., 2] * vn + k[..., 3] * vt) / DT
            e = e + 0.5 * (self.fw * area * dens).sum()
        return e

    def residual(self, d):
        u = self.full(d).requires_grad_(True)
        g, = torch.autograd.grad(self.potential(u), u)
        g = g.detach().index_add(0, self.pf.reshape(-1), self.pressure((self.X + u.detach())[self.pf]).reshape(-1, 3))
        return g[self.free].reshape(-1)

    def product(self, d, x):
        """K x by differentiating the residual once more."""
        u = self.full(d).requires_grad_(True)
        v = self.full(x)
        g, = torch.autograd.grad(self.potential(u), u, create_graph=True)
        h, = torch.autograd.grad((g * v).sum(), u)
        _, dp = torch.func.jvp(self.pressure, ((self.X + u.detach())[self.pf],), (v[self.pf],))
        return h.index_add(0, self.pf.reshape(-1), dp.reshape(-1, 3))[self.free].reshape(-1)

    def element_tangents(self, d, chunk):
        u = self.full(d)[self.elems]
        hess = torch.func.vmap(torch.func.hessian(self.energy), chunk_size=chunk)
        k = hess(u, self.G, self.R, self.wd)
        xf = (self.X + self.full(d))[self.pf]
        return k, torch.func.vmap(torch.func.jacfwd(self.pressure))(xf)

    def solve(self, d, b):
        """K^-1 b by block elimination over the breadth-first levels of the
        mesh's node graph (blocks couple to their neighbours only)."""
        K, Kp = self.element_tangents(d, 256)
        n_nodes = len(self.X)
        free = self.free.cpu().numpy()
        of = -np.ones(n_nodes, dtype=np.int64)
        of[free] = np.arange(len(free))
        lists = [self.elems.cpu().numpy(), self.pf.cpu().numpy()]
        # levels: from the nodes at the low end of the longest extent
        Xn = self.X.cpu().numpy()
        ax = int(np.argmax(np.ptp(Xn, axis=0)))
        lev = -np.ones(n_nodes, dtype=np.int64)
        lev[Xn[:, ax] <= Xn[:, ax].min() + 1e-9 * np.ptp(Xn[:, ax])] = 0
        el = lists[0]
        k = 0
        while (lev < 0).any():
            touched = np.unique(el[(lev[el] == k).any(axis=1)])
            touched = touched[lev[touched] < 0]
            k += 1
            lev[touched] = k
        lf = lev[free]
        order = np.argsort(lf, kind="stable")
        sizes = np.bincount(lf, minlength=k + 1)
        pos = np.empty(len(free), dtype=np.int64)
        start = np.concatenate([[0], np.cumsum(sizes)])
        pos[order] = np.arange(len(free)) - start[lf[order]]
        blocks = [[torch.zeros(3 * sizes[i], 3 * sizes[j], dtype=F64, device="cuda") if 0 <= j <= k else None
                   for j in (i - 1, i, i + 1)] for i in range(k + 1)]
        of_t, lf_t, pos_t = (torch.as_tensor(a, device="cuda") for a in (of, lf, pos))
        comp = torch.arange(3, device="cuda")
        for nodes, mats in ((self.elems, K), (self.pf, Kp)):
            f = of_t[nodes]
            ia, ib = f[:, :, None].expand(-1, -1, f.shape[1]), f[:, None, :].expand(-1, f.shape[1], -1)
            keep = (ia >= 0) & (ib >= 0)
            ia, ib = ia[keep], ib[keep]
            vals = mats.permute(0, 1, 3, 2, 4)[keep]
            la, lb = lf_t[ia], lf_t[ib]
            for i in range(k + 1):
                at = la == i
                for o in (-1, 0, 1):
                    m = at & (lb == i + o)
                    if not bool(m.any()):
                        continue
                    B = blocks[i][o + 1]
                    rows = 3 * pos_t[ia[m]][:, None, None] + comp[None, :, None]
                    cols = 3 * pos_t[ib[m]][:, None, None] + comp[None, None, :]
                    B.view(-1).index_add_(0, (rows * B.shape[1] + cols).reshape(-1), vals[m].reshape(-1))
        dof = [torch.as_tensor((3 * order[start[i]:start[i + 1]][:, None] + np.arange(3)).reshape(-1), device="cuda")
               for i in range(k + 1)]
        ys, Us = [], []
        for i in range(k + 1):
            D, rhs = blocks[i][1], b[dof[i]]
            if i:
                D = D - blocks[i][0] @ Us[-1]
                rhs = rhs - blocks[i][0] @ ys[-1]
            right = rhs[:, None] if i == k else torch.cat([blocks[i][2], rhs[:, None]], dim=1)
            sol = torch.linalg.solve(D, right)
            Us.append(sol[:, :-1])
            ys.append(sol[:, -1])
            blocks[i] = [None, None, None]
        x = torch.empty_like(b)
        for i in range(k, -1, -1):
            if i < k:
                ys[i] = ys[i] - Us[i] @ ys[i + 1]
            x[dof[i]] = ys[i]
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("precond", "apply"):
        return None  # a preconditioner's action: defined by its own construction alone
    s = _inputs(case, seed)
    n = len(s["d"])
    if kind in ("newton", "gmres") and n > 100000:
        return None  # a direct solve takes minutes
    plain = _Plain(s, case)
    if kind == "residual":
        return plain.residual(s["d"])
    if kind == "spmv":
        return plain.product(s["d"], s["x"])
    if kind == "tangent":
        return plain.residual(s["d"]), plain.product(s["d"], s["x"])
    delta = plain.solve(s["d"], -plain.residual(s["d"]))
    return s["d"] + delta if kind == "newton" else delta
