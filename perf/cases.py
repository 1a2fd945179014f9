"""Performance cases of the solver: what a user's program calls, over the sizes it is used at.

Kinds of case (``kind``):

* ``gauss``    return mapping of every Gauss point at a displacement increment, from a committed state;
* ``tangent``  a Newton linearisation by hand: assemble the tangent and the residual, apply K and K^+;
* ``dual``     the dual operators of a user's own Krylov method on an assembled tangent: F, P_N and the
               preconditioner (with its second projection);
* ``solve``    one dual solve (Algorithm 3) on an assembled tangent, FP64 or mixed precision;
* ``ramp``     load steps of the semismooth Newton method from the zero state, one load case or several at once
               (each on a context and stream of its own).

Meshes: ``n``^3 bricks on the unit cube in ``parts``^3 equal boxes (``parts`` > 0), or in a seeded uneven
partition into boxes of 4..12 elements per edge (``parts`` = 0, ``cut_seed``).  Boundary conditions and material
are those of the repository's workloads (u = 0 on z = 0, traction on z = 1).

``exact`` restates the outputs in plain torch FP64: its own mesh, gluing matrix and material law, dense factors of
the boxes, a dense coarse matrix, and conjugate gradients on the undecomposed problem.
"""
import math
import random

import numpy as np
import torch

import paper_1205_1926_gb300 as T
import workloads as W

F64 = torch.float64
DEV = "cuda"
MATERIAL = {"young": 206900.0, "poisson": 0.29, "sigma_y": 450.0, "hardening": 10000.0}


# ---------------------------------------------------------------------------- cases
def _case(name, kind, n, parts, **kw):
    c = {"name": name, "kind": kind, "n": n, "parts": parts, "cut_seed": 0, "precond": "lumped", "mixed": False}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the material law on eight small boxes, as a user checks a model with (launches and latency)
        _case("gauss_12", "gauss", 12, 2, dtan=False),
        # the material law alone at the largest mesh one load case is run on, and with the consistent tangent
        # returned to the caller (a user's own assembly) at the profiling size
        _case("gauss_96", "gauss", 96, 12, dtan=False),
        _case("gauss_48_dtan", "gauss", 48, 6, dtan=True),
        # linearisation with refactorised boxes: a quarter of the boxes yielding, and the uneven partition
        _case("tangent_48_plastic", "tangent", 48, 6, hot=54),
        # operators of a user's own Krylov method: the timed mesh with some boxes yielding; a coarse problem
        # large enough for the plane solver
        _case("dual_64_plastic", "dual", 64, 8, hot=24),
        _case("dual_96", "dual", 96, 12, hot=0),
        # one dual solve in the default precision (elastic first solve of a load step) at the timed size, with the
        # Dirichlet preconditioner on a mesh of small boxes, and in mixed precision on the uneven partition
        _case("solve_64_fp64", "solve", 64, 8, hot=0, rtol=1e-11),
        _case("solve_32_dirichlet", "solve", 32, 4, hot=4, precond="dirichlet", rtol=1e-11),
        _case("solve_40_uneven_mixed", "solve", 40, 0, cut_seed=1, hot=4, mixed=True, rtol=1e-11),
        # load histories: the paper-sized small body in FP64; the headline setting (mixed precision, history and
        # learned start) at the timed size; four load directions at once
        _case("ramp_12_fp64", "ramp", 12, 2, steps=3, history=0, learned=False, n_cases=1, ntol=1e-10, rtol=1e-12),
        _case("ramp_64_learned", "ramp", 64, 8, steps=20, history=7, learned=True, n_cases=1, mixed=True, ntol=1e-10,
              rtol=1e-11),
        _case("ramp_48_four_cases", "ramp", 48, 6, steps=3, history=8, learned=False, n_cases=4, mixed=True,
              ntol=1e-10, rtol=1e-11),
    ]


def draw(rng):
    kind = rng.choice(("gauss", "tangent", "dual", "solve", "solve", "ramp", "ramp"))
    uneven = kind != "gauss" and rng.random() < 0.3
    if uneven:
        hi = {"tangent": 40, "dual": 48, "solve": 40, "ramp": 24}[kind]
        n, parts, cut = rng.randint(20, hi), 0, rng.randint(1, 1000)
    else:
        # boxes of a edges of elements each, b boxes per axis: odd boxes and odd counts among them
        hi = {"gauss": 96, "tangent": 48, "dual": 72, "solve": 56, "ramp": 48}[kind]
        n = int(round(math.exp(rng.uniform(math.log(10), math.log(hi)))))
        a = rng.choice((5, 6, 7, 8, 8, 8, 9))
        parts, cut = max(2, int(round(n / a))), 0
        n = min(a * parts, hi // a * a)
        parts = n // a
    c = {"kind": kind, "n": n, "parts": parts, "cut_seed": cut, "precond": "lumped", "mixed": False}
    boxes = parts ** 3 if parts else 27
    if kind == "gauss":
        c["dtan"] = n <= 56 and rng.random() < 0.5
    elif kind in ("tangent", "dual"):
        c["hot"] = rng.randint(0, max(1, min(54, boxes // 6)))
    elif kind == "solve":
        c["mixed"] = rng.random() < 0.5 or (uneven and n > 28)
        c["hot"] = rng.randint(0, max(1, min(8, boxes // 8)))
        c["rtol"] = 1e-11
        if not c["mixed"] and not uneven and n <= 32 and rng.random() < 0.3:
            c["precond"] = "dirichlet"
    else:
        c["mixed"] = uneven or n > 32 or rng.random() < 0.6
        c["history"] = 7 if uneven else rng.choice((0, 4, 7))
        c["learned"] = bool(c["mixed"] and c["history"] == 7 and rng.random() < 0.7)
        c["n_cases"] = rng.choice((1, 1, 2)) if c["mixed"] and not uneven else 1
        c["steps"] = 2 if uneven else rng.randint(2, 4)
        c["ntol"], c["rtol"] = 1e-10, 1e-11
    return c


def _cuts(case):
    n, parts = case["n"], case["parts"]
    if parts:
        c = tuple(i * (n // parts) for i in range(parts + 1))
        return (c, c, c)
    return W.irregular_cube(n, case["cut_seed"]).cuts


def _workload(case):
    n = case["n"]
    return W.Workload(name="perf_%d_%d" % (n, case["parts"]), nel=(n, n, n), cuts=_cuts(case))


# ---------------------------------------------------------------------------- inputs
def _rand(gen, *shape):
    return torch.randn(*shape, generator=gen, dtype=F64, device=DEV)


def _box_starts(case):
    """First decomposed dof of every box (x-fastest order), and the total."""
    cx, cy, cz = _cuts(case)
    off = [0]
    for k in range(len(cz) - 1):
        for j in range(len(cy) - 1):
            for i in range(len(cx) - 1):
                off.append(off[-1] + 3 * (cx[i + 1] - cx[i] + 1) * (cy[j + 1] - cy[j] + 1) * (cz[k + 1] - cz[k] + 1))
    return off


def _state_inputs(case, gen, n_gp):
    """A committed state as a loaded body has it: stresses of a fraction of the yield stress, some hardening."""
    return 100.0 * _rand(gen, 6, n_gp), 1e-3 * torch.rand(n_gp, generator=gen, dtype=F64, device=DEV)


def _increment(case, gen, seed):
    """Displacement increment that is far below yield except in ``hot`` boxes, where about half the points yield."""
    off = _box_starts(case)
    h = 1.0 / case["n"]
    du = _rand(gen, off[-1]) * (1e-5 * h)
    rng = random.Random(seed)
    for p in rng.sample(range(len(off) - 1), min(case["hot"], len(off) - 1)):
        du[off[p]:off[p + 1]] *= 120.0
    return du


def _traction_load(ctx, t):
    f = torch.zeros(ctx.sizes["n_dof"], dtype=F64, device=DEV)
    ctx.traction_load(t, f)
    return f


def _directions(case, seed):
    """One traction direction per load case in the x-y plane, and its size as a multiple of first yield."""
    rng = random.Random(1000 + seed)
    k = case["n_cases"]
    th = rng.uniform(0.0, 2.0 * math.pi)
    return [((math.cos(th + 2.0 * math.pi * i / k), math.sin(th + 2.0 * math.pi * i / k), 0.0),
             rng.uniform(1.3, 1.5)) for i in range(k)]


def _solve_inputs(case, seed):
    """Increment of the linearisation, and the load: a traction and small body forces."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    du = _increment(case, gen, seed)
    body = _rand(gen, du.numel()) * (1e-3 / case["n"] ** 2)
    th = random.Random(seed).uniform(0.0, 2.0 * math.pi)
    return du, body, (math.cos(th), math.sin(th), 0.3)


def prepare(case, seed):
    kw = {"precond": T.PRECOND_DIRICHLET} if case["precond"] == "dirichlet" else {}
    several = case.get("n_cases", 1) > 1
    ctx = T.Context(_workload(case), stream=torch.cuda.Stream() if several else None, **kw)
    nd, ng, m = ctx.sizes["n_dof"], ctx.sizes["n_gp"], ctx.sizes["n_mult"]
    if case["mixed"]:
        ctx.set_precision(True, 1e-4)
    new = lambda *s, t=F64: torch.zeros(*s, dtype=t, device=DEV)  # noqa: E731
    s = {"case": case, "ctx": ctx}
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if case["kind"] == "gauss":
        sig, kap = _state_inputs(case, gen, ng)
        ctx.set_state(sigma=sig, kappa=kap)
        s["du"] = _rand(gen, nd) * (1e-3 / case["n"])
        s["out"] = [new(6, ng), new(ng), new(ng, t=torch.uint8)] + ([new(21, ng)] if case["dtan"] else [])
    elif case["kind"] == "tangent":
        s["du"] = _increment(case, gen, seed)
        s["df"] = _rand(gen, nd) * (1.0 / case["n"] ** 2)
        s["x"] = _rand(gen, nd)
        s["out"] = [new(nd), new(nd), new(nd)]
    elif case["kind"] == "dual":
        ctx.assemble_tangent(_increment(case, gen, seed), new(nd))
        s["x"] = _rand(gen, m)
        s["out"] = [new(m) for _ in range(4)]
    elif case["kind"] == "solve":
        du, body, t = _solve_inputs(case, seed)
        ctx.assemble_tangent(du, new(nd))
        s["f"] = _traction_load(ctx, t) + body
        s["out"] = [new(nd), new(m)]
    else:
        ctxs, fulls = [ctx], []
        if several:
            torch.cuda.synchronize()
            for _ in range(case["n_cases"] - 1):
                ctxs.append(T.Context(_workload(case), stream=torch.cuda.Stream(), **kw))
                if case["mixed"]:
                    ctxs[-1].set_precision(True, 1e-4)
        for t, factor in _directions(case, seed):
            t_y = ctx.first_yield_traction(t, case["rtol"])
            f = torch.zeros(nd, dtype=F64, device=DEV)
            torch.cuda.synchronize()
            ctx.traction_load(tuple(factor * t_y * v for v in t), f)
            torch.cuda.synchronize()
            fulls.append(f / case["steps"])
        s["ctxs"], s["dfs"] = ctxs, fulls
        s["zero"] = [new(nd), new(6, ng), new(ng)]
        s["out"] = [[new(nd), new(6, ng), new(ng)] for _ in ctxs]
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------- one pass
def run(s):
    case, ctx = s["case"], s["ctx"]
    if case["kind"] == "gauss":
        out = s["out"]
        ctx.return_map(s["du"], out[0], out[1], out[2], out[3] if case["dtan"] else None)
        return out
    if case["kind"] == "tangent":
        f, kx, kdx = s["out"]
        ctx.assemble_tangent(s["du"], s["df"], f)
        ctx.apply("K", s["x"], kx)
        ctx.apply("kdag", s["x"], kdx)
        return [f, kx, kdx]
    if case["kind"] == "dual":
        fx, w, z, y = s["out"]
        ctx.apply("F", s["x"], fx)
        ctx.apply("projector", s["x"], w)
        ctx.apply("precond", w, z)
        ctx.apply("projector", z, y)
        return [fx, w, z, y]
    if case["kind"] == "solve":
        u, lam = s["out"]
        ctx.dual_pcg(s["f"], u, lam, rtol=case["rtol"], maxit=5000)
        return [u, lam]
    # load steps from the zero state with a fresh history, as a program that starts a load history does
    zu, zs, zk = s["zero"]
    for c in s["ctxs"]:
        c.set_state(u=zu, sigma=zs, kappa=zk)
        c.set_learned(False)
        c.set_recycling(case["history"])
        if case["learned"]:
            c.set_learned(True)
    for _ in range(case["steps"]):
        if len(s["ctxs"]) == 1:
            ctx.time_step(s["dfs"][0], case["ntol"], case["rtol"])
        else:
            T.time_step_cases(s["ctxs"], s["dfs"], case["ntol"], case["rtol"])
    for c, (u, sig, kap) in zip(s["ctxs"], s["out"]):
        c.get_state(u=u, sigma=sig, kappa=kap)
    return s["out"]


# ---------------------------------------------------------------------------- work
def _box_counts(case):
    cx, cy, cz = ([b - a for a, b in zip(c, c[1:])] for c in _cuts(case))
    return [(a, b, c) for c in cz for b in cy for a in cx]


def work(case):
    """Bytes and operations one pass cannot do without: inputs read and outputs written once, the operations of
    the method on the boxes' band factors (the sparsest form of K^+ the method prescribes)."""
    boxes = _box_counts(case)
    nd = sum(3 * (a + 1) * (b + 1) * (c + 1) for a, b, c in boxes)
    ng = 8 * case["n"] ** 3
    ni = sum(3 * ((a + 1) * (b + 1) * (c + 1) - max(0, a - 1) * max(0, b - 1) * max(0, c - 1)) for a, b, c in boxes)
    m = ni // 2 + 1
    shapes = {b: 3 * (b[0] + 1) * (b[1] + 1) * (b[2] + 1) * (3 * (b[0] + 1) * (b[1] + 2) + 3) for b in boxes}
    solve = sum(4.0 * shapes[b] for b in boxes)               # one K^+ apply on every box
    factors = 8.0 * sum(shapes.values())                       # one factor per shape
    gauss_b, gauss_f = 8.0 * (nd + 7 * ng + 7 * ng) + ng, 160.0 * ng
    if case["kind"] == "gauss":
        return {"bytes": gauss_b + (8.0 * 21 * ng if case["dtan"] else 0.0), "flops": gauss_f}
    refac = 0.0
    if case.get("hot"):
        b = boxes[len(boxes) // 2]
        refac = case["hot"] * shapes[b] * float(3 * (b[0] + 1) * (b[1] + 2) + 3)
    if case["kind"] == "tangent":
        return {"bytes": 8.0 * (nd * 6 + 7 * ng) + factors, "flops": gauss_f + 100.0 * ng + 2 * solve + refac}
    if case["kind"] == "dual":
        return {"bytes": 8.0 * 9 * m + factors + 8.0 * 36 * len(boxes) ** 2, "flops": solve + 4.0 * 81 * ni}
    its = 30.0                                                 # iterations of a typical dual solve
    if case["kind"] == "solve":
        return {"bytes": 8.0 * (2 * nd + m) + factors, "flops": its * solve}
    steps = case["steps"] * case["n_cases"]                    # each with about three Newton iterations
    return {"bytes": 8.0 * steps * (2 * nd + 7 * ng) + factors, "flops": 3.0 * steps * (its * solve + gauss_f)}


# ---------------------------------------------------------------------------- the same in plain FP64 torch
_OFF = np.array([[0, 0, 0], [1, 0, 0], [1, 1, 0], [0, 1, 0], [0, 0, 1], [1, 0, 1], [1, 1, 1], [0, 1, 1]])
_PAIRS = [(i, j) for i in range(6) for j in range(i, 6)]


def _t(a, dtype=None):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device=DEV)


class _Body:
    """Decomposed cube in plain arrays: boxes, elements, gluing and Dirichlet rows, material."""

    def __init__(self, case):
        n = self.n = case["n"]
        cuts = _cuts(case)
        self.h = 1.0 / n
        lam = MATERIAL["young"] * MATERIAL["poisson"] / ((1 + MATERIAL["poisson"]) * (1 - 2 * MATERIAL["poisson"]))
        self.mu = MATERIAL["young"] / (2 * (1 + MATERIAL["poisson"]))
        self.H, self.sy = MATERIAL["hardening"], MATERIAL["sigma_y"]
        C = np.zeros((6, 6))
        C[:3, :3] = lam
        C[range(3), range(3)] += 2 * self.mu
        C[range(3, 6), range(3, 6)] = self.mu
        self.C = _t(C)
        dev = np.diag([1.0, 1, 1, 0.5, 0.5, 0.5])
        dev[:3, :3] -= 1.0 / 3.0
        self.Edev = _t(dev)                                     # strain -> deviatoric strain in stress form
        # strain matrices of the eight Gauss points
        B = np.zeros((8, 6, 24))
        for g in range(8):
            xi = np.array([2 * (g & 1) - 1, 2 * (g >> 1 & 1) - 1, 2 * (g >> 2) - 1]) / math.sqrt(3.0)
            for a in range(8):
                s = 2 * _OFF[a] - 1
                v = 1 + s * xi
                d = s / 8.0 * np.array([v[1] * v[2], v[0] * v[2], v[0] * v[1]]) * 2.0 / self.h
                c = 3 * a
                B[g, 0, c], B[g, 1, c + 1], B[g, 2, c + 2] = d
                B[g, 3, c], B[g, 3, c + 1] = d[1], d[0]
                B[g, 4, c + 1], B[g, 4, c + 2] = d[2], d[1]
                B[g, 5, c], B[g, 5, c + 2] = d[2], d[0]
        self.B = _t(B)
        self.w = self.h ** 3 / 8.0
        self.Kel = self.w * torch.einsum("gia,ij,gjb->ab", self.B, self.C, self.B)
        # boxes: local nodes, elements
        self.boxes, gnode, edofs, off = [], [], [], 0
        N1 = n + 1
        for K in range(len(cuts[2]) - 1):
            for J in range(len(cuts[1]) - 1):
                for I in range(len(cuts[0]) - 1):
                    o = np.array([cuts[0][I], cuts[1][J], cuts[2][K]])
                    d = np.array([cuts[0][I + 1], cuts[1][J + 1], cuts[2][K + 1]]) - o
                    nn = d + 1
                    lk, lj, li = np.meshgrid(np.arange(nn[2]), np.arange(nn[1]), np.arange(nn[0]), indexing="ij")
                    li, lj, lk = li.ravel(), lj.ravel(), lk.ravel()
                    gnode.append((li + o[0]) + N1 * ((lj + o[1]) + N1 * (lk + o[2])))
                    e = (li < d[0]) & (lj < d[1]) & (lk < d[2])
                    ln = np.stack([(li[e] + a[0]) + nn[0] * ((lj[e] + a[1]) + nn[1] * (lk[e] + a[2])) for a in _OFF], 1)
                    ld = (3 * ln[:, :, None] + np.arange(3)).reshape(-1, 24)
                    fix = [0, 1, 2, 3 * d[0] + 1, 3 * d[0] + 2, 3 * nn[0] * d[1] + 2]
                    xyz = (np.stack([li, lj, lk], 1) - d / 2.0) * self.h
                    self.boxes.append({"off": off, "n": 3 * len(li), "dims": tuple(d), "ld": ld, "fix": fix,
                                       "e0": sum(len(x) for x in edofs), "xyz": xyz})
                    edofs.append(ld + off)
                    off += 3 * len(li)
        self.nd = off
        self.edof = _t(np.concatenate(edofs))                   # [elements][24] decomposed dofs
        gnode = np.concatenate(gnode)
        self.gnode = gnode
        # rows of B: (global node, component) order, copies in box order
        order = np.argsort(gnode, kind="stable")
        nodes, start, k = np.unique(gnode[order], return_index=True, return_counts=True)
        clamped = nodes // (N1 * N1) == 0                       # z = 0: all components fixed
        nrow = np.where(clamped, k, k - 1)
        row0 = np.concatenate([[0], np.cumsum(3 * nrow)])[:-1]
        rows, cols, vals = [], [], []
        for c in range(3):
            for kk in range(1, 9):
                s = np.flatnonzero((k == kk) & clamped)
                for j in range(kk):
                    rows.append(row0[s] + c * kk + j)
                    cols.append(3 * order[start[s] + j] + c)
                    vals.append(np.ones(len(s)))
                s = np.flatnonzero((k == kk) & ~clamped)
                for r in range(1, kk):
                    for j in range(r + 1):
                        rows.append(row0[s] + c * (kk - 1) + r - 1)
                        cols.append(3 * order[start[s] + j] + c)
                        vals.append(np.full(len(s), (1.0 if j < r else -float(r)) / math.sqrt(r * (r + 1.0))))
        self.m = int(3 * nrow.sum())
        self.brow, self.bcol, self.bval = (_t(np.concatenate(v)) for v in (rows, cols, vals))
        self.gdof = _t((3 * gnode[:, None] + np.arange(3)).ravel())
        self.ng = 3 * N1 ** 3
        self.free = torch.ones(self.ng, dtype=F64, device=DEV)
        self.free[:3 * N1 * N1] = 0.0

    # B, B^T and the undecomposed vector
    def Bx(self, v):
        return torch.zeros(self.m, dtype=F64, device=DEV).index_add_(0, self.brow, self.bval * v[self.bcol])

    def BTx(self, x):
        return torch.zeros(self.nd, dtype=F64, device=DEV).index_add_(0, self.bcol, self.bval * x[self.brow])

    def glue(self, v):
        return torch.zeros(self.ng, dtype=F64, device=DEV).index_add_(0, self.gdof, v) * self.free

    def traction(self, t):
        """Uniform traction on z = 1, a quarter of each element face to each of its nodes, in the owning box."""
        f = torch.zeros(self.nd, dtype=F64, device=DEV)
        for b in self.boxes:
            e = np.arange(len(b["ld"]))
            d = b["dims"]
            if round(b["xyz"][-1, 2] / self.h * 2) != d[2] or self.gnode[b["off"] // 3 + b["n"] // 3 - 1] // (self.n + 1) ** 2 != self.n:
                continue
            top = b["ld"][e // (d[0] * d[1]) == d[2] - 1][:, 12:].ravel()
            val = np.tile(np.array(t) * self.h ** 2 / 4.0, len(top) // 3)
            f.index_add_(0, _t(top + b["off"]), _t(val))
        return f

    # material at Gauss points: strains [E][8][6], state [E][8][..]
    def strains(self, du):
        return torch.einsum("gia,ea->egi", self.B, du[self.edof])

    def law(self, eta, sig, kap, tangent=False):
        """dsigma, dkappa, plastic flag (and, for plastic points, a, b, n of T = C - a Edev - b n n^T)."""
        ds = eta @ self.C
        tau = sig + ds
        p = tau[..., :3].mean(-1, keepdim=True)
        dv = torch.cat([tau[..., :3] - p, tau[..., 3:]], -1)
        nrm = (dv[..., :3].square().sum(-1) + 2.0 * dv[..., 3:].square().sum(-1)).sqrt()
        y = self.sy + self.H * kap
        phi = math.sqrt(1.5) * nrm - y
        pl = phi > 1e-12 * y
        phi = torch.where(pl, phi, torch.zeros_like(phi))
        nh = dv / nrm.clamp_min(1e-300)[..., None]
        c = 3 * self.mu / (3 * self.mu + self.H)
        ds = ds - (c * math.sqrt(2.0 / 3.0) * phi)[..., None] * nh
        if not tangent:
            return ds, phi / (3 * self.mu + self.H), pl
        rho = math.sqrt(2.0 / 3.0) * y / nrm.clamp_min(1e-300)
        a = torch.where(pl, 2 * self.mu * c * (1 - rho), torch.zeros_like(rho))
        b = torch.where(pl, 2 * self.mu * c * rho, torch.zeros_like(rho))
        return ds, phi / (3 * self.mu + self.H), pl, a, b, nh

    def force(self, ds):
        fe = self.w * torch.einsum("gia,egi->ea", self.B, ds)
        return torch.zeros(self.nd, dtype=F64, device=DEV).index_add_(0, self.edof.ravel(), fe.ravel())

    def linearise(self, du, sig=None, kap=None):
        """Residual stresses and the element corrections of the tangent at du."""
        E = self.edof.shape[0]
        sig = torch.zeros(E, 8, 6, dtype=F64, device=DEV) if sig is None else sig
        kap = torch.zeros(E, 8, dtype=F64, device=DEV) if kap is None else kap
        ds, dk, pl, a, b, nh = self.law(self.strains(du), sig, kap, True)
        self.pe = torch.nonzero(pl.any(1)).ravel()
        D = a[self.pe][..., None, None] * self.Edev + b[self.pe][..., None, None] * nh[self.pe][..., :, None] * nh[self.pe][..., None, :]
        DB = torch.einsum("egij,gjb->egib", D, self.B)
        self.dK = self.w * torch.einsum("gia,egib->eab", self.B, DB)
        return ds, dk

    def Kx(self, x):
        xe = x[self.edof]
        ye = xe @ self.Kel
        if len(self.pe):
            ye[self.pe] -= torch.einsum("eab,eb->ea", self.dK, xe[self.pe])
        return torch.zeros(self.nd, dtype=F64, device=DEV).index_add_(0, self.edof.ravel(), ye.ravel())

    def _factor(self, b, dK=None):
        n = b["n"]
        ld = _t(b["ld"])
        K = torch.zeros(n * n, dtype=F64, device=DEV)
        Ke = self.Kel.expand(len(b["ld"]), 24, 24)
        if dK is not None:
            Ke = Ke.clone()
            Ke[dK[0]] -= dK[1]
        K.index_add_(0, (ld[:, :, None] * n + ld[:, None, :]).ravel(), Ke.reshape(-1))
        K = K.view(n, n)
        fix = _t(np.array(b["fix"]))
        K[fix, :] = 0.0
        K[:, fix] = 0.0
        K[fix, fix] = 1.0
        return torch.linalg.cholesky(K), fix

    def kdag(self, x):
        """K^+ x box by box (fixing dofs removed), dense factors; elastic boxes of one shape together."""
        y = torch.zeros_like(x)
        pe = self.pe.cpu().numpy()
        el = {}
        for b in self.boxes:
            lo, hi = np.searchsorted(pe, [b["e0"], b["e0"] + len(b["ld"])])
            if hi == lo:
                el.setdefault(b["dims"], []).append(b)
                continue
            L, fix = self._factor(b, (_t(pe[lo:hi] - b["e0"]), self.dK[lo:hi]))
            y[b["off"]:b["off"] + b["n"]] = self._apply(L, fix, x[b["off"]:b["off"] + b["n"], None])[:, 0]
        for bs in el.values():
            L, fix = self._factor(bs[0])
            idx = _t(np.stack([np.arange(b["off"], b["off"] + b["n"]) for b in bs], 1))
            y[idx] = self._apply(L, fix, x[idx])
        return y

    @staticmethod
    def _apply(L, fix, X):
        X = X.clone()
        X[fix] = 0.0
        Y = torch.cholesky_solve(X, L)
        Y[fix] = 0.0
        return Y

    def projector(self):
        """x -> x - G^T (G G^T)^-1 G x with G = R^T B^T, R the boxes' rigid-body modes (any basis)."""
        R = np.zeros((self.nd, 6))
        box = np.zeros(self.nd, dtype=np.int64)
        for p, b in enumerate(self.boxes):
            r = np.zeros((b["n"], 6))
            X = b["xyz"]
            for c in range(3):
                r[c::3, c] = 1.0
            r[1::3, 3], r[2::3, 3] = -X[:, 2], X[:, 1]
            r[0::3, 4], r[2::3, 4] = X[:, 2], -X[:, 0]
            r[0::3, 5], r[1::3, 5] = -X[:, 1], X[:, 0]
            R[b["off"]:b["off"] + b["n"]] = np.linalg.qr(r)[0]
            box[b["off"]:b["off"] + b["n"]] = p
        R, box = _t(R), _t(box)
        l = 6 * len(self.boxes)
        # G^T as (row, box) pairs with six values, then G G^T from the pairs of each row
        key, inv = torch.unique(self.brow * len(self.boxes) + box[self.bcol], return_inverse=True)
        val = torch.zeros(len(key), 6, dtype=F64, device=DEV).index_add_(0, inv, self.bval[:, None] * R[self.bcol])
        row, bx = key // len(self.boxes), key % len(self.boxes)
        GGT = torch.zeros(l * l, dtype=F64, device=DEV)
        first = torch.searchsorted(row, torch.arange(self.m, device=DEV))
        last = torch.searchsorted(row, torch.arange(self.m, device=DEV), right=True)
        six = torch.arange(6, device=DEV)
        for i in range(8):
            for j in range(8):
                r = torch.nonzero((last - first > i) & (last - first > j)).ravel()
                if not len(r):
                    continue
                a, b = first[r] + i, first[r] + j
                at = (6 * bx[a][:, None, None] + six[:, None]) * l + 6 * bx[b][:, None, None] + six
                GGT.index_add_(0, at.ravel(), (val[a][:, :, None] * val[b][:, None, :]).ravel())
        L = torch.linalg.cholesky(GGT.view(l, l))

        def apply(x):
            g = torch.zeros(len(self.boxes), 6, dtype=F64, device=DEV).index_add_(0, bx, val * x[row][:, None])
            h = torch.cholesky_solve(g.reshape(-1, 1), L).view(-1, 6)
            return x - torch.zeros(self.m, dtype=F64, device=DEV).index_add_(0, row, (val * h[bx]).sum(1))

        return apply

    def solve(self, f, du0=None):
        """Undecomposed displacement of the linearised problem by conjugate gradients (Jacobi), decomposed."""
        diag = torch.diagonal(self.Kel).expand(len(self.edof), 24).clone()
        if len(self.pe):
            diag[self.pe] -= torch.diagonal(self.dK, dim1=1, dim2=2)
        D = torch.zeros(self.nd, dtype=F64, device=DEV).index_add_(0, self.edof.ravel(), diag.ravel())
        D = self.glue(D) + (1.0 - self.free)
        A = lambda v: self.glue(self.Kx(v[self.gdof]))  # noqa: E731
        x, r = torch.zeros(self.ng, dtype=F64, device=DEV), self.glue(f)
        x, r = self._cg(A, D, x, r, 1e-14)
        r = self.glue(f) - A(x)                                  # one refinement from the true residual
        dx, _ = self._cg(A, D, torch.zeros_like(x), r, 1e-6)
        return (x + dx)[self.gdof]

    @staticmethod
    def _cg(A, D, x, r, tol):
        z = r / D
        p, rz, r0 = z, torch.dot(r, z), torch.dot(r, r / D)
        for it in range(20000):
            Ap = A(p)
            al = rz / torch.dot(p, Ap)
            x, r = x + al * p, r - al * Ap
            z = r / D
            new = torch.dot(r, z)
            if it % 20 == 0 and not float(new) > tol * tol * float(r0):
                break
            p, rz = z + (new / rz) * p, new
        return x, r


def exact(case, seed):
    if case["kind"] == "ramp" and (case["n"] > 12 or case["n_cases"] > 1):
        return None                                              # Newton histories by plain CG take minutes
    b = _Body(case)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    E = b.edof.shape[0]
    soa = lambda a: a.reshape(8 * E, -1).T.contiguous()  # noqa: E731
    if case["kind"] == "gauss":
        sig, kap = _state_inputs(case, gen, 8 * E)
        du = _rand(gen, b.nd) * (1e-3 / case["n"])
        out = [torch.empty(6, 8 * E, dtype=F64, device=DEV), torch.empty(8 * E, dtype=F64, device=DEV),
               torch.empty(8 * E, dtype=torch.uint8, device=DEV)]
        if case["dtan"]:
            out.append(torch.empty(21, 8 * E, dtype=F64, device=DEV))
        eta_all, step = b.edof, 1 << 16
        for e in range(0, E, step):
            s = slice(8 * e, min(8 * E, 8 * (e + step)))
            eta = torch.einsum("gia,ea->egi", b.B, du[eta_all[e:e + step]]).reshape(-1, 6)
            ds, dk, pl, a, bb, nh = b.law(eta, sig[:, s].T, kap[s], True)
            out[0][:, s], out[1][s], out[2][s] = ds.T, dk, pl.to(torch.uint8)
            if case["dtan"]:
                D = b.C - a[:, None, None] * b.Edev - bb[:, None, None] * nh[:, :, None] * nh[:, None, :]
                for k, (i, j) in enumerate(_PAIRS):
                    out[3][k, s] = D[:, i, j]
        return out
    if case["kind"] == "tangent":
        du = _increment(case, gen, seed)
        df = _rand(gen, b.nd) * (1.0 / case["n"] ** 2)
        x = _rand(gen, b.nd)
        ds, _ = b.linearise(du)
        return [df - b.force(ds), b.Kx(x), b.kdag(x)]
    if case["kind"] == "dual":
        b.linearise(_increment(case, gen, seed))
        x = _rand(gen, b.m)
        P = b.projector()
        w = P(x)
        z = b.Bx(b.Kx(b.BTx(w)))
        return [b.Bx(b.kdag(b.BTx(x))), w, z, P(z)]
    if case["kind"] == "solve":
        du, body, t = _solve_inputs(case, seed)
        b.linearise(du)
        f = b.traction(t) + body
        u = b.solve(f)
        return [u, b.Bx(f - b.Kx(u))]
    # load steps of the undecomposed body, Newton to stagnation
    (t, factor), = _directions(case, seed)
    sig, kap = torch.zeros(E, 8, 6, dtype=F64, device=DEV), torch.zeros(E, 8, dtype=F64, device=DEV)
    u = torch.zeros(b.nd, dtype=F64, device=DEV)
    f1 = b.traction(t)
    b.linearise(u)
    ds = b.law(b.strains(b.solve(f1)), sig, kap)[0]
    p = ds[..., :3].mean(-1, keepdim=True)
    dv = torch.cat([ds[..., :3] - p, ds[..., 3:]], -1)
    q = math.sqrt(1.5) * float((dv[..., :3].square().sum(-1) + 2 * dv[..., 3:].square().sum(-1)).max().sqrt())
    df = f1 * (factor * b.sy / q / case["steps"])
    for _ in range(case["steps"]):
        du = torch.zeros_like(u)
        for _ in range(12):
            ds, dk = b.linearise(du, sig, kap)
            d = b.solve(df - b.force(ds))
            du = du + d
            if float(d.norm()) <= 1e-13 * float(du.norm()):
                break
        ds, dk, _ = b.law(b.strains(du), sig, kap)
        u, sig, kap = u + du, sig + ds, kap + dk
    return [[u, soa(sig), kap.reshape(-1)]]
