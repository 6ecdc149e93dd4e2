"""The calls by which the speed of this framework is judged, over the range it is used in.

Elements from a few hundred (one small body: latency and launches) to about half a million (a cantilever that fills
the GPU); the four element types, straight-sided and curved; FP32 and FP64 element math; both laws, with and without
damping; the atomic and the deterministic scatter; force, operator product, both in one call, the adjoint, a
differentiable forward and backward, and whole implicit steps. Every number is random from the seed; `exact` computes
the same outputs in 64 bits with plain torch.
"""
import functools
import itertools
import math
import random

import numpy as np
import torch

from paper_2602_17002_gb300 import autograd, tlfe

EDGE = 0.05                                # cell edge (m)
NPE = {"T4": 4, "T10": 10, "H8": 8, "Q27": 27}
CODE = {"T4": tlfe.T4, "T10": tlfe.T10, "H8": tlfe.H8, "Q27": tlfe.Q27}
RULES = {"T4": (1,), "T10": (4, 5), "H8": (8,), "Q27": (27,)}
PER_CELL = {"T4": 6, "T10": 6, "H8": 1, "Q27": 1}
MU, LAM, ETA, RHO = 3.8e6, 5.8e6, 1e3, 1000.0
STEP, GRAVITY = 1e-3, (0.0, 0.0, -9.81)
NEWTON = dict(newton_rtol=1e-10, cg_rtol=1e-4, max_newton=12, max_cg=2000)


def _case(op, elem, nq, cells, law="nh", damped=False, fp=32, scatter="atomic", curved=False, bodies=1, tuned=False,
          name=None):
    c = dict(op=op, elem=elem, nq=nq, nx=cells[0], ny=cells[1], nz=cells[2], law=law, damped=damped, fp=fp,
             scatter=scatter, curved=curved, bodies=bodies, tuned=tuned)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest model of the test-suite: 384 quadratic tetrahedra in FP64, one force and one tangent product,
        # as a static solve of a small part asks for them; launches and latency
        _case("force_product", "T10", 4, (4, 4, 4), law="svk", fp=64, name="block_384_t10_fp64"),
        # a small damped beam in a time loop: force, operator product and adjoint of 480 elements
        _case("step", "T10", 5, (20, 2, 2), damped=True, name="beam_480_t10"),
        # the benchmark's cantilever: 480,000 quadratic tetrahedra, damped; force, operator product and adjoint
        _case("step", "T10", 5, (200, 20, 20), damped=True, tuned=True, name="beam_480k_t10"),
        # the same operations in plain FP64, the reference path and the residuals of implicit steps
        _case("step", "T10", 5, (100, 10, 10), damped=True, fp=64, name="beam_60k_t10_fp64"),
        # many bodies of uneven size, element type and law in one mesh, tuned once: force and tangent product
        _case("force_product", "mixed", 0, (40, 40, 40), bodies=40, tuned=True, name="batch_40_mixed"),
        # parameter identification: per-element (mu, lambda), a loss on the force, forward and backward
        _case("learn", "T10", 5, (40, 39, 41), damped=True, name="learn_384k_t10"),
        # implicit steps of eight clamped beams under gravity, to a tight residual: Newton, Jacobi-PCG
        _case("newton", "T10", 5, (40, 8, 8), bodies=8, name="newton_8_beams_t10"),
        # a block of bricks with odd cell counts: tangent product alone, as an outer Krylov solver calls it
        _case("product", "H8", 8, (61, 53, 47), law="svk", name="block_152k_h8"),
        # the triquadratic brick
        _case("step", "Q27", 27, (67, 19, 21), damped=True, name="beam_27k_q27"),
        # curved (isoparametric) quadratic tetrahedra: the reference gradients are streamed
        _case("step", "T10", 5, (36, 31, 29), damped=True, curved=True, name="curved_194k_t10"),
        # the deterministic scatter, as a run that has to repeat bit for bit uses it
        _case("step", "T10", 5, (100, 20, 20), damped=True, scatter="sorted", name="sorted_240k_t10"),
        # explicit dynamics on linear tetrahedra: the force alone
        _case("force", "T4", 1, (59, 51, 47), name="block_849k_t4"),
    ]


# elements of the largest draw of each operation, so that a drawn case costs no more than the largest listed one
MOST = {"force": 480_000, "product": 480_000, "force_product": 480_000, "step": 480_000, "learn": 380_000}
SHARE = {"T4": 1.0, "T10": 1.0, "H8": 0.4, "Q27": 0.055}     # elements of that type of about the same work


def draw(rng):
    if rng.random() < 0.12:
        n = rng.randint(2, 7)
        return _case("newton", "T10", 5, (rng.randint(9, 37), n, n), bodies=rng.randint(1, 8))
    if rng.random() < 0.12:
        n = rng.randint(12, 40)
        return _case("force_product", "mixed", 0, (n, n, n), bodies=rng.randint(5, 40), tuned=rng.random() < 0.5)
    op = rng.choice(["force", "product", "force_product", "step", "step", "learn"])
    elem = "T10" if op == "learn" else rng.choice(["T4", "T10", "T10", "H8", "Q27"])
    fp = 32 if op == "learn" else rng.choice([32, 32, 32, 64])
    most = MOST[op] * SHARE[elem] * (0.06 if fp == 64 else 1.0)
    n = math.exp(rng.uniform(math.log(360 * min(1.0, 4 * SHARE[elem])), math.log(most))) / PER_CELL[elem]
    a, b = math.exp(rng.uniform(0.0, 1.6)), math.exp(rng.uniform(-0.2, 0.2))      # long beams to near cubes
    ny = max(2, round((n / a) ** (1 / 3) * b))
    nz = max(2, round((n / a) ** (1 / 3) / b))
    nx = max(2, math.floor(n / (ny * nz)))
    curved = elem in ("T10", "H8") and op != "learn" and rng.random() < 0.2
    return _case(op, elem, rng.choice(RULES[elem]), (nx, ny, nz), law=rng.choice(["nh", "svk"]),
                 damped=rng.random() < 0.5, fp=fp, scatter=rng.choice(["atomic", "atomic", "sorted"]),
                 curved=curved, tuned=rng.random() < 0.3)


# ---- meshes ----------------------------------------------------------------

def _corners():
    """The six tetrahedra of a cell around its main diagonal: corner offsets, positively oriented."""
    out = []
    for perm in itertools.permutations(range(3)):
        p = np.zeros((4, 3), np.int64)
        for k, ax in enumerate(perm):
            p[k + 1:, ax] += 1
        if np.linalg.det((p[1:] - p[0]).astype(float)) < 0:
            p[[2, 3]] = p[[3, 2]]
        out.append(p)
    return out


@functools.lru_cache(maxsize=4)
def _box(elem, nx, ny, nz):
    """(X, conn) of a box of nx x ny x nz cells; T10 and Q27 live on the half-step grid."""
    s = 2 if elem in ("T10", "Q27") else 1
    g = (s * nx + 1, s * ny + 1, s * nz + 1)
    X = np.stack(np.meshgrid(*(np.arange(m) * (EDGE / s) for m in g[::-1]), indexing="ij")[::-1], -1).reshape(-1, 3)
    cell = np.stack(np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")[::-1], -1).reshape(-1, 3)
    base = s * (cell[:, 0] + g[0] * (cell[:, 1] + g[1] * cell[:, 2]))
    if elem in ("T4", "T10"):
        offs = []
        for p in _corners():
            o = [s * q for q in p]
            if elem == "T10":
                o += [p[a] + p[b] for a, b in ((0, 1), (1, 2), (0, 2), (0, 3), (1, 3), (2, 3))]
            offs += o
    else:
        m = 2 if elem == "H8" else 3
        offs = [np.array([i, j, k]) for k in range(m) for j in range(m) for i in range(m)]
    off = np.array([o[0] + g[0] * (o[1] + g[1] * o[2]) for o in offs])
    conn = (base[:, None] + off[None, :]).reshape(-1, NPE[elem]).astype(np.int32)
    return np.ascontiguousarray(X), conn


def _plan(case):
    """The bodies of a case: (element type, points, cells, law, mu, lam). The batch's are uneven, fixed by the case."""
    if case["elem"] != "mixed":
        return [(case["elem"], case["nq"], (case["nx"], case["ny"], case["nz"]), case["law"], MU, LAM)] * case["bodies"]
    r, out = random.Random(case["bodies"]), []
    for _ in range(case["bodies"]):
        elem = r.choice(["T4", "T10", "H8"])
        ne = math.exp(r.uniform(math.log(1e3), math.log(3.0 * case["nx"] ** 3)))       # elements, log-uniform
        n = max(1, round((ne / PER_CELL[elem]) ** (1 / 3)))
        E, nu = math.exp(r.uniform(math.log(1e6), math.log(1e9))), r.uniform(0.2, 0.45)
        out.append((elem, RULES[elem][-1], (n, n, max(1, round(ne / PER_CELL[elem] / n ** 2))), r.choice(["nh", "svk"]),
                    E / (2 * (1 + nu)), E * nu / ((1 + nu) * (1 - 2 * nu))))
    return out


@functools.lru_cache(maxsize=2)
def _topology(items):
    """(X, blocks [(elem, nq, conn, body)], bodies [(law, mu, lam)]) of a case."""
    case = dict(items)
    Xs, per, mats, off = [], {}, [], 0
    for b, (elem, nq, cells, law, mu, lam) in enumerate(_plan(case)):
        X, conn = _box(elem, *cells)
        per.setdefault((elem, nq), []).append((conn + np.int32(off), b))
        Xs.append(X)
        mats.append((law, mu, lam))
        off += X.shape[0]
    blocks = [(elem, nq, np.concatenate([c for c, _ in v]), np.concatenate([np.full(len(c), b, np.int32) for c, b in v]))
              for (elem, nq), v in per.items()]
    return np.concatenate(Xs), blocks, mats


def _key(case):
    return tuple(sorted((k, v) for k, v in case.items() if k != "name"))


def _inputs(case, seed):
    """Everything random, on the GPU: reference nodes, displacement (a bending field and noise), velocities,
    directions, parameters."""
    X, blocks, mats = _topology(_key(case))
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = X.shape[0]

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64) * 2 - 1

    dt = torch.float64 if case["fp"] == 64 else torch.float32
    Xd = torch.from_numpy(X).cuda()
    if case["curved"]:
        Xd = Xd + 0.04 * EDGE * uniform(n, 3)
    d = dict(X=Xd, blocks=blocks, mats=mats)
    if case["elem"] == "mixed":            # each body stretched at random, 1 % noise
        u = torch.empty(n, 3, device="cuda", dtype=torch.float64)
        S = uniform(len(mats), 3, 3) * 0.025
        node_body = np.zeros(n, np.int64)
        for _, _, conn, body in blocks:
            node_body[conn] = body[:, None]
        S = (S + S.transpose(1, 2))[torch.from_numpy(node_body).cuda()]
        u = torch.einsum("nab,nb->na", S, Xd) + 0.01 * EDGE * uniform(n, 3)
    else:                                  # cantilever bending by 5 % of the length at most, 0.1 % noise
        L = float(X[:, 0].max())
        tip = (0.02 if case["op"] == "newton" else 0.05) * L * (0.7 + 0.3 * float(uniform(1)))
        x, z = Xd[:, 0], Xd[:, 2] - 0.5 * float(X[:, 2].max())
        u = torch.stack([-z * tip * 3 * x * (2 * L - x) / (2 * L ** 3), torch.zeros_like(x),
                         tip * x * x * (3 * L - x) / (2 * L ** 3)], 1)
        u += (1e-5 if case["op"] == "newton" else 1e-3) * EDGE * uniform(n, 3)
    d["u"] = u
    d["udot"] = (0.01 * normal(n, 3)).to(dt) if case["damped"] else None
    d["v"] = normal(n, 3).to(dt)
    d["cot"] = normal(n, 3).to(dt)
    if case["op"] == "learn":              # log-parameters in 32 bits, as an optimiser holds them
        ne = blocks[0][2].shape[0]
        d["u"] = u.float()
        d["p"] = (0.25 * normal(ne, 2) + torch.tensor([math.log(4e6), math.log(6e6)], device="cuda",
                                                      dtype=torch.float64)).float()
        p_true = d["p"].double() + 0.05 * normal(ne, 2)
        d["target"] = _force(case, dict(d, u=d["u"].double()), torch.exp(p_true)).float()
    if case["op"] == "newton":
        d["v0"] = 1e-3 * normal(n, 3)
        d["fixed"] = (Xd[:, 0] < 1e-9).to(torch.uint8)
    return d


# ---- the calls ---------------------------------------------------------------

def prepare(case, seed):
    d = _inputs(case, seed)
    code = {"svk": tlfe.SVK, "nh": tlfe.NEOHOOKE}
    mesh = tlfe.Mesh(d["X"].cpu().numpy(), [(CODE[e], nq, conn, body) for e, nq, conn, body in d["blocks"]],
                     [(code[law], mu, lam, ETA if case["damped"] else 0.0, 0.0, RHO) for law, mu, lam in d["mats"]],
                     precision=tlfe.FP64 if case["fp"] == 64 else tlfe.FP32,
                     scatter=tlfe.SCATTER_SORTED if case["scatter"] == "sorted" else tlfe.SCATTER_ATOMIC)
    s = dict(case=case, mesh=mesh, ac=1.0 if case["damped"] else 0.0)
    for k in ("u", "udot", "v", "cot", "p", "target", "v0", "fixed"):
        if k in d:
            s[k] = d[k]
    if case["tuned"]:
        mesh.autotune(s["u"].double(), s["udot"], s["v"])
    if case["op"] == "learn":
        for k in ("u", "udot", "p"):
            if s[k] is not None:
                s[k].requires_grad_(True)
    s["f"], s["y"] = (torch.empty_like(s["v"]) for _ in range(2))
    return s


def run(s):
    op, m = s["case"]["op"], s["mesh"]
    if op == "force":
        return m.internal_force(s["u"], s["udot"], out=s["f"])
    if op == "product":
        return m.tangent_matvec(s["u"], s["udot"], s["v"], 0.0, 1.0, s["ac"], out=s["y"])
    if op == "force_product":
        return m.force_matvec(s["u"], s["udot"], s["v"], 0.0, 1.0, s["ac"], f=s["f"], y=s["y"])
    if op == "step":
        f, y = m.force_matvec(s["u"], s["udot"], s["v"], 0.0, 1.0, s["ac"], f=s["f"], y=s["y"])
        gu, gud, _ = m.vjp(s["u"], s["udot"], s["cot"], want_udot=s["udot"] is not None, want_theta=False)
        return [f, y, gu] + ([gud] if gud is not None else [])
    if op == "learn":
        for k in ("u", "udot", "p"):
            if s[k] is not None:
                s[k].grad = None
        f = autograd.internal_force(m, s["u"], s["udot"], torch.exp(s["p"]).double())
        loss = 0.5 * (f - s["target"]).square().sum()
        loss.backward()
        return [f.detach(), loss.detach(), s["u"].grad, s["p"].grad] + ([] if s["udot"] is None else [s["udot"].grad])
    v, report = m.newton_step(s["u"], s["v0"], STEP, GRAVITY, fixed=s["fixed"], **NEWTON)
    if report["code"] != 0:
        raise RuntimeError("the step did not converge: %r" % (report,))
    return v, torch.add(s["u"], v, alpha=STEP)


# What cannot be done without, by element: connectivity and reference nodes read once, each node array once; per point
# and field the 3x3 gradient of a nodal field (J^{-1}: 45 multiply-adds or more), per point the stress, its derivative
# or its adjoint.
POINT = {"force": (1, 1, 300), "product": (2, 1, 650), "force_product": (2, 2, 650), "step": (4, 4, 1300),
         "learn": (2, 3, 950), "newton": (2, 1, 650)}      # gathered fields, scattered fields, flops of the law


def work(case):
    X, blocks, _ = _topology(_key(case))
    n, b = X.shape[0], 8 if case["fp"] == 64 else 4
    elems = sum(c.shape[0] for _, _, c, _ in blocks)
    points = sum(c.shape[0] * nq for _, nq, c, _ in blocks)
    conn = sum(c.size for _, _, c, _ in blocks) * 4
    nin, nout, law = POINT[case["op"]]
    visc = 1 if case["damped"] else 0
    state = n * (24 + 24 + visc * 3 * b)
    calls = {"step": 2, "learn": 2}.get(case["op"], 1)
    out = {"force": 1, "product": 2, "force_product": 3, "step": 4 + visc + 1, "learn": 4 + visc, "newton": 4}[case["op"]]
    nbytes = calls * (conn + state) + n * 3 * b * out + (elems * 24 if case["op"] == "learn" else 0)
    flops = points * (law * (1 + 0.4 * visc) + 90 * (nin + nout + visc * (2 if calls == 2 else 1)))
    if case["op"] == "newton":             # an operator product and its vectors per CG iteration, some tens of them
        nbytes, flops = 60 * nbytes, 60 * flops
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits, by plain torch ---------------------------------------

@functools.lru_cache(maxsize=None)
def _rule(elem, nq):
    """Points, weights, shape functions (q, i) and their parent gradients (q, i, k)."""
    if elem in ("T4", "T10"):
        if nq == 1:
            L, w = [[0.25] * 4], [1 / 6]
        elif nq == 4:
            a, b = (5 + 3 * math.sqrt(5)) / 20, (5 - math.sqrt(5)) / 20
            L, w = [[a if j == q else b for j in range(4)] for q in range(4)], [1 / 24] * 4
        elif nq == 5:
            L = [[0.25] * 4] + [[0.5 if j == q else 1 / 6 for j in range(4)] for q in range(4)]
            w = [-2 / 15] + [3 / 40] * 4
        else:                              # collapsed Gauss rule, exact to degree 5
            x, gw = np.polynomial.legendre.leggauss(4)
            x, gw, L, w = (x + 1) / 2, gw / 2, [], []
            for (a, wa), (b, wb), (c, wc) in itertools.product(zip(x, gw), repeat=3):
                p = (a, b * (1 - a), c * (1 - a) * (1 - b))
                L.append([1 - sum(p), *p])
                w.append(wa * wb * wc * (1 - a) ** 2 * (1 - b))
        return np.array(L)[:, 1:], np.array(w)
    x, gw = np.polynomial.legendre.leggauss(2 if nq == 8 else 3)
    pts = [(a[0], b[0], c[0], a[1] * b[1] * c[1]) for c in zip(x, gw) for b in zip(x, gw) for a in zip(x, gw)]
    return np.array(pts)[:, :3], np.array(pts)[:, 3]


def _shapes(elem, xi):
    """s_i and d s_i / d xi_k at the points xi (q, 3)."""
    if elem in ("T4", "T10"):
        L = np.concatenate([1 - xi.sum(1, keepdims=True), xi], 1)
        dL = np.array([[-1.0, -1, -1], [1, 0, 0], [0, 1, 0], [0, 0, 1]])
        if elem == "T4":
            return L, np.broadcast_to(dL, (len(xi), 4, 3)).copy()
        e = ((0, 1), (1, 2), (0, 2), (0, 3), (1, 3), (2, 3))
        s = np.concatenate([L * (2 * L - 1), np.stack([4 * L[:, a] * L[:, b] for a, b in e], 1)], 1)
        g = [(4 * L[:, i] - 1)[:, None] * dL[i] for i in range(4)]
        g += [4 * (L[:, b][:, None] * dL[a] + L[:, a][:, None] * dL[b]) for a, b in e]
        return s, np.stack(g, 1)
    if elem == "H8":
        l1, d1 = (lambda x: [(1 - x) / 2, (1 + x) / 2]), (lambda x: [-0.5 + 0 * x, 0.5 + 0 * x])
    else:
        l1, d1 = (lambda x: [x * (x - 1) / 2, 1 - x * x, x * (x + 1) / 2]), (lambda x: [x - 0.5, -2 * x, x + 0.5])
    l, d = [l1(xi[:, k]) for k in range(3)], [d1(xi[:, k]) for k in range(3)]
    idx = [(i, j, k) for k in range(len(l[0])) for j in range(len(l[0])) for i in range(len(l[0]))]
    s = np.stack([l[0][i] * l[1][j] * l[2][k] for i, j, k in idx], 1)
    g = np.stack([np.stack([d[0][i] * l[1][j] * l[2][k], l[0][i] * d[1][j] * l[2][k], l[0][i] * l[1][j] * d[2][k]], 1)
                  for i, j, k in idx], 1)
    return s, g


def _cof(F):
    a, b, c = F[..., 0, :], F[..., 1, :], F[..., 2, :]
    return torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], -2)


def _element_force(h, w, law, mu, lam, eta, ue, ude):
    """f_e = sum_q w P(F, Fdot) h: h (e, q, i, 3), w (e, q); mu, lam (e,)."""
    eye = torch.eye(3, device="cuda", dtype=torch.float64)
    F = torch.einsum("eia,eqib->eqab", ue, h) + eye
    mu, lam = mu[:, None, None, None], lam[:, None, None, None]
    if law == "svk":
        E = 0.5 * (F.transpose(-1, -2) @ F - eye)
        P = F @ (lam * E.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] * eye + 2 * mu * E)
    else:
        C = _cof(F)
        J = (F * C).sum((-1, -2), keepdim=True) / 3
        P = mu * J ** (-2 / 3) * (F - (F * F).sum((-1, -2), keepdim=True) / 3 * C / J)
        P = P + (lam + 2 * mu / 3) * (J - 1) * C
    if ude is not None:
        A = torch.einsum("eia,eqib->eqab", ude, h).transpose(-1, -2) @ F
        P = P + F @ (eta * (A + A.transpose(-1, -2)))
    return torch.einsum("eq,eqab,eqib->eia", w, P, h)


def _pieces(case, d, theta=None, most=1 << 19):
    """The elements in pieces of one law: (connectivity, h, w, force(ue, ude, mu, lam), mu, lam, first element)."""
    base = 0
    for elem, nq, conn, body in d["blocks"]:
        xi, wq = _rule(elem, nq)
        g, wq = torch.from_numpy(_shapes(elem, xi)[1]).cuda(), torch.from_numpy(wq).cuda()
        conn_d = torch.from_numpy(conn).cuda().long()
        laws = np.array([d["mats"][b][0] == "svk" for b in range(len(d["mats"]))])[body]
        mu0, lam0 = (torch.tensor([m[k] for m in d["mats"]], device="cuda", dtype=torch.float64) for k in (1, 2))
        for law, which in (("nh", ~laws), ("svk", laws)):
            ids = torch.from_numpy(np.flatnonzero(which)).cuda()
            for at in ids.split(max(1, most // nq)):
                if at.numel() == 0:
                    continue
                cn = conn_d[at]
                Jm = torch.einsum("eia,qib->eqab", d["X"][cn], g)
                det = torch.linalg.det(Jm)
                h = torch.einsum("qib,eqba->eqia", g, torch.linalg.inv(Jm))
                bd = torch.from_numpy(body).cuda()[at].long()
                mu, lam = (mu0[bd], lam0[bd]) if theta is None else (theta[at, 0], theta[at, 1])
                yield cn, functools.partial(_element_force, h, wq * det, law, eta=ETA), mu, lam, at + base
        base += conn.shape[0]


def _at(x, cn):
    return None if x is None else x[cn].double()


def _force(case, d, theta=None):
    f = torch.zeros_like(d["X"])
    for cn, fe, mu, lam, _ in _pieces(case, d, theta):
        f.index_add_(0, cn.reshape(-1), fe(mu=mu, lam=lam, ue=_at(d["u"], cn), ude=_at(d["udot"], cn)).reshape(-1, 3))
    return f


def _product(case, d, v, aK, aC, pieces=None):
    y = torch.zeros_like(d["X"])
    for cn, fe, mu, lam, _ in pieces if pieces is not None else _pieces(case, d):
        ue, ude, ve = _at(d["u"], cn), _at(d["udot"], cn), _at(v, cn)
        if ude is None:
            ye = torch.func.jvp(lambda a: fe(mu=mu, lam=lam, ue=a, ude=None), (ue,), (aK * ve,))[1]
        else:
            ye = torch.func.jvp(lambda a, b: fe(mu=mu, lam=lam, ue=a, ude=b), (ue, ude), (aK * ve, aC * ve))[1]
        y.index_add_(0, cn.reshape(-1), ye.reshape(-1, 3))
    return y


def _adjoint(case, d, cot, theta=None):
    gu, gud = torch.zeros_like(d["X"]), torch.zeros_like(d["X"])
    gth = torch.zeros(sum(c.shape[0] for _, _, c, _ in d["blocks"]), 2, device="cuda", dtype=torch.float64)
    for cn, fe, mu, lam, at in _pieces(case, d, theta):
        a = [t.detach().requires_grad_(True) for t in (_at(d["u"], cn), mu, lam)]
        b = None if d["udot"] is None else _at(d["udot"], cn).requires_grad_(True)
        got = torch.autograd.grad(fe(mu=a[1], lam=a[2], ue=a[0], ude=b), a + ([] if b is None else [b]), _at(cot, cn))
        gu.index_add_(0, cn.reshape(-1), got[0].reshape(-1, 3))
        gth[at, 0], gth[at, 1] = got[1], got[2]
        if b is not None:
            gud.index_add_(0, cn.reshape(-1), got[3].reshape(-1, 3))
    return gu, gud, gth


def _mass(d):
    """M x of the consistent mass matrix, by the elements' own shape functions."""
    parts = []
    for elem, nq, conn, _ in d["blocks"]:
        xi, wq = _rule(elem, 64)
        s, g = (torch.from_numpy(t).cuda() for t in _shapes(elem, xi))
        cn = torch.from_numpy(conn).cuda().long()
        det = torch.linalg.det(torch.einsum("eia,ib->eab", d["X"][cn], g[0]))     # straight-sided elements
        hat = torch.einsum("q,qi,qj->ij", torch.from_numpy(wq).cuda(), s, s)
        parts.append((cn, RHO * det[:, None, None], hat))

    def apply(x):
        y = torch.zeros_like(x)
        for cn, c, hat in parts:
            y.index_add_(0, cn.reshape(-1), (c * torch.einsum("ij,eja->eia", hat, x[cn])).reshape(-1, 3))
        return y
    return apply


def _newton(case, d):
    """The backward-Euler velocity by Newton and conjugate gradients, well below the tolerance of the call."""
    M, free = _mass(d), (d["fixed"] == 0).double()[:, None]
    grav = M(torch.tensor(GRAVITY, device="cuda", dtype=torch.float64).expand_as(d["X"]).contiguous())
    v, first = d["v0"] * free, None
    for _ in range(10):
        e = dict(d, u=d["u"] + STEP * v, udot=None)
        g = free * (M(v - d["v0"]) / STEP + _force(case, e) - grav)
        norm = float(g.norm())
        first = first or norm
        if norm <= 3e-13 * first:
            break
        pieces = list(_pieces(case, e))
        x, r = torch.zeros_like(v), -g
        p, rr = r.clone(), float((r * r).sum())
        stop = rr * 1e-12
        for _ in range(3000):
            q = free * (M(p) / STEP + _product(case, e, p, STEP, 0.0, pieces))
            a = rr / float((p * q).sum())
            x, r = x + a * p, r - a * q
            rr, old = float((r * r).sum()), rr
            if rr <= stop:
                break
            p = r + (rr / old) * p
        v = v + x
    return v


def exact(case, seed):
    d, op, ac = _inputs(case, seed), case["op"], 1.0 if case["damped"] else 0.0
    if op == "force":
        return _force(case, d)
    if op == "product":
        return _product(case, d, d["v"], 1.0, ac)
    if op == "force_product":
        return _force(case, d), _product(case, d, d["v"], 1.0, ac)
    if op == "step":
        gu, gud, _ = _adjoint(case, d, d["cot"])
        return [_force(case, d), _product(case, d, d["v"], 1.0, ac), gu] + ([gud] if case["damped"] else [])
    if op == "learn":
        d["u"] = d["u"].double()
        theta = torch.exp(d["p"].double())
        f = _force(case, d, theta)
        r = f - d["target"].double()
        gu, gud, gth = _adjoint(case, d, r, theta)
        return [f, 0.5 * r.square().sum(), gu, gth * theta] + ([gud] if case["damped"] else [])
    v = _newton(case, d)
    return v, d["u"] + STEP * v
