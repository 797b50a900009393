"""The work this library is used for, as cases to be timed and compared.

listed() names the cases, draw() gives more of the same ranges, prepare()
makes what a program has in hand before the call, run() is one pass through
the public entry points, work() is what a pass cannot do without and exact()
is the same result in 64 bits from plain torch and numpy.

Kinds of case:
  apply    v = A u on the finest (DG) level of a box mesh, FP64 or FP32
  hex      v = A u on an unstructured hexahedral mesh
  smooth   five Chebyshev-Jacobi steps on the DG level or the FE level below it
  solve    flexible CG with the V-cycle to 1e-10, cycle in FP64 or FP32
  multi    the same for several right-hand sides of one problem at once
  batch    the same for several unequal problems at once
"""
import math
from functools import lru_cache

import numpy as np
import torch

from paper_1910_01900_gb300 import Batch, Context
from paper_1910_01900_gb300.native import create_unstructured

STEPS = 5          # smoothing steps of the default cycle
RTOL = 1e-10       # relative residual of the solves


def listed():
    return [
        # outer residual of a curved FP64 solve: the operator of a time step or Krylov iteration
        dict(name="apply_f64_curved16_k5", kind="apply", prec=0, deform=1, m0=16, m1=16, m2=16, k=5),
        # operator throughput on a large deformed mesh in the cycle's precision
        dict(name="apply_f32_curved42_k5", kind="apply", prec=1, deform=1, m0=42, m1=42, m2=42, k=5),
        # the same on a large box at high degree
        dict(name="apply_f32_cube32_k7", kind="apply", prec=1, deform=0, m0=32, m1=32, m2=32, k=7),
        # general hexahedra (a mesh generator's output): the operator alone
        dict(name="apply_f32_hex15_k3", kind="hex", prec=1, m0=15, m1=13, m2=14, k=3),
        # post-smoothing on a curved DG level with odd sizes
        dict(name="smooth_f32_dg_curved21_k3", kind="smooth", level="dg", prec=1, deform=1, m0=21, m1=20, m2=19, k=3),
        # post-smoothing on the continuous level below the DG level of the 32^3 cube
        dict(name="smooth_f32_fe_cube32_k4", kind="smooth", level="fe", prec=1, deform=0, m0=32, m1=32, m2=32, k=4),
        # the smallest solve in use, bound by latency and launches
        dict(name="solve_mixed_cube4_k3", kind="solve", prec=1, deform=0, m0=4, m1=4, m2=4, k=3),
        # mixed-precision solve on a deformed mesh
        dict(name="solve_mixed_curved16_k5", kind="solve", prec=1, deform=1, m0=16, m1=16, m2=16, k=5),
        # mixed-precision solve on the large cube
        dict(name="solve_mixed_cube32_k4", kind="solve", prec=1, deform=0, m0=32, m1=32, m2=32, k=4),
        # the same in FP64 throughout (the benchmark's default)
        dict(name="solve_f64_cube32_k4", kind="solve", prec=0, deform=0, m0=32, m1=32, m2=32, k=4),
        # many right-hand sides of one problem
        dict(name="multi32_mixed_cube16_k4", kind="multi", nrhs=32, prec=1, deform=0, m0=16, m1=16, m2=16, k=4),
        # many unequal problems
        dict(name="batch16_mixed", kind="batch", prec=1,
             problems="20:2 22:4 20:3 8:5 18:2 10:5 12:4 14:3 24:6 16:2 8:6 10:2 14:5 18:4 22:2 12:6"),
    ]


def draw(rng):
    """One more case: every kind, degrees 1..8, equal and unequal sides, odd sizes."""

    def sides(k, lo, hi, even=False):
        dofs = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = dofs ** (1 / 3) / (k + 1)
        out = []
        for _ in range(3):
            s = max(2, round(side * rng.uniform(0.85, 1.1)))
            if even:
                s = max(4, 2 * round(s / 2))
            out.append(int(s))
        return dict(m0=out[0], m1=out[1], m2=out[2])

    kind = rng.choice(["apply", "apply", "apply", "hex", "smooth", "smooth", "solve", "solve", "multi", "batch"])
    deform, prec = rng.randrange(2), rng.randrange(2)
    if kind == "apply":
        k = rng.randint(1, 8)
        return dict(kind=kind, prec=prec, deform=deform, k=k, **sides(k, 2e3, 1.5e7 if prec else 3e6))
    if kind == "hex":
        k = rng.randint(1, 6)
        return dict(kind=kind, prec=prec, k=k, **sides(k, 5e3, 4e5))
    if kind == "smooth":
        k = rng.randint(2, 8)
        return dict(kind=kind, level=rng.choice(["dg", "fe"]), prec=1, deform=deform, k=k, **sides(k, 5e4, 3e6, even=True))
    if kind == "solve":
        k = rng.randint(2, 7)
        return dict(kind=kind, prec=rng.choice([0, 1, 1]), deform=deform, k=k, **sides(k, 6e3, 1.5e6, even=True))
    if kind == "multi":
        k, nrhs = rng.randint(2, 5), rng.randint(2, 24)
        return dict(kind=kind, nrhs=nrhs, prec=1, deform=deform, k=k, **sides(k, 8e3, 7e6 / nrhs, even=True))
    some = ["%d:%d" % (2 * rng.randint(4, 9), rng.randint(2, 5)) for _ in range(rng.randint(3, 12))]
    return dict(kind=kind, prec=1, problems=" ".join(some))


# ------------------------------------------------------------------ the calls

_kept = {}   # the newest case's context: a program builds it once and keeps it
_stream = []


def stream():
    if not _stream:
        _stream.append(torch.cuda.Stream())
    return _stream[0]


def _sizes(case):
    return (case["m0"], case["m1"], case["m2"])


def _problems(case):
    return [dict(m=int(p.split(":")[0]), k=int(p.split(":")[1])) for p in case["problems"].split()]


def _context(case):
    key = tuple(sorted((a, b) for a, b in case.items() if a != "name"))
    if _kept.get("key") != key:
        _kept.clear()
        s = stream()
        if case["kind"] == "hex":
            V, C, _, _ = _hex_mesh(*_sizes(case))
            ctx = create_unstructured(V, C, case["k"], stream=s)
        elif case["kind"] == "batch":
            ctx = Batch(_problems(case), precision=case["prec"], stream=s)
        else:
            ctx = Context(_sizes(case), case["k"], deform=case["deform"], precision=case["prec"],
                          operator_only=case["kind"] == "apply", stream=s)
        _kept.update(key=key, ctx=ctx)
    return _kept["ctx"]


def _uniform(n, seed, dtype, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return torch.rand(n, generator=g, dtype=dtype, device=device) * 2 - 1


def _dtype(prec):
    return torch.float32 if prec else torch.float64


def _dofs(case):
    n3 = (case["k"] + 1) ** 3
    if case.get("level") == "fe":
        return math.prod(m * case["k"] + 1 for m in _sizes(case))
    return math.prod(_sizes(case)) * n3


def _inputs(case, seed, device="cuda"):
    """The vectors of a pass, from the seed alone: uniform values, as residuals and search directions have every frequency."""
    kind = case["kind"]
    if kind in ("apply", "hex"):
        return dict(u=_uniform(_dofs(case), seed, _dtype(case["prec"]), device))
    if kind == "smooth":
        n, t = _dofs(case), _dtype(case["prec"])
        return dict(b=_uniform(n, seed, t, device), x0=_uniform(n, seed + 7919, t, device))
    if kind == "solve":
        return dict(b=_uniform(_dofs(case), seed, torch.float64, device))
    if kind == "multi":
        return dict(b=_uniform(case["nrhs"] * _dofs(case), seed, torch.float64, device).view(case["nrhs"], -1))
    return dict(b=[_uniform(p["m"] ** 3 * (p["k"] + 1) ** 3, seed + 7919 * i, torch.float64, device)
                   for i, p in enumerate(_problems(case))])


def prepare(case, seed):
    s = dict(_inputs(case, seed), case=case, ctx=_context(case))
    first = s.get("u", s.get("b"))
    s["out"] = [torch.zeros_like(t) for t in first] if isinstance(first, list) else torch.zeros_like(first)
    return s


def run(state):
    case, ctx, out = state["case"], state["ctx"], state["out"]
    kind = case["kind"]
    with torch.cuda.stream(stream()):
        if kind in ("apply", "hex"):
            ctx.apply(state["u"], out)
        elif kind == "smooth":
            out.copy_(state["x0"])
            ctx.smooth(ctx.num_levels - (1 if case["level"] == "dg" else 2), state["b"], out, STEPS)
        elif kind == "solve":
            out.zero_()
            ctx.solve(state["b"], out, rtol=RTOL)
        elif kind == "multi":
            out.zero_()
            ctx.solve_multi(state["b"], out, rtol=RTOL)
        else:
            for x in out:
                x.zero_()
            ctx.solve(state["b"], out, rtol=RTOL)
    return out


def _apply_work(dofs, cells, k, deform, size):
    """One operator application: the vector in and out, a deformed cell's mapping nodes (new ones per cell: 27 points); 1D
    products (7 where the operator is a sum of three tensor products, else 12) and the face terms."""
    n = k + 1
    return dict(bytes=2 * size * dofs + (27 * 3 * 8 * cells if deform else 0),
                flops=dofs * (2 * n * (12 if deform else 7) + 24))


def work(case):
    if case["kind"] == "batch":
        every = [work(dict(kind="solve", prec=case["prec"], deform=0, m0=p["m"], m1=p["m"], m2=p["m"], k=p["k"]))
                 for p in _problems(case)]
        return {key: sum(w[key] for w in every) for key in ("bytes", "flops")}
    size, deform = 4 if case["prec"] else 8, case.get("deform", 1)
    cells = math.prod(_sizes(case))
    one = _apply_work(_dofs(case), cells, case["k"], deform, size)
    if case["kind"] in ("apply", "hex"):
        return one
    if case["kind"] == "smooth":   # b, x and the inverse diagonal in, x out
        return dict(bytes=4 * size * _dofs(case) + one["bytes"] - 2 * size * _dofs(case), flops=STEPS * one["flops"])
    # about six iterations, each ten applications on the DG level and ten on the FE level of the same degree, and one outside
    n = case.get("nrhs", 1)
    return dict(bytes=n * 16 * _dofs(case) + one["bytes"] - 2 * size * _dofs(case), flops=n * 6 * 18 * one["flops"])


# ------------------------------------------------- the same in 64 bits, plainly

def _lobatto(n):
    """n Gauss-Lobatto points on [0, 1]."""
    if n == 2:
        return np.array([0.0, 1.0])
    inner = np.polynomial.legendre.Legendre.basis(n - 1).deriv().roots()
    return (np.concatenate([[-1.0], np.sort(np.real(inner)), [1.0]]) + 1) / 2


def _lagrange(nodes, pts):
    """Values and derivatives of the Lagrange basis: two matrices [point][basis]."""
    n = len(nodes)
    V, D = np.ones((len(pts), n)), np.zeros((len(pts), n))
    for j in range(n):
        others = [i for i in range(n) if i != j]
        for i in others:
            V[:, j] *= (pts - nodes[i]) / (nodes[j] - nodes[i])
            t = np.full(len(pts), 1.0 / (nodes[j] - nodes[i]))
            for l in others:
                if l != i:
                    t *= (pts - nodes[l]) / (nodes[j] - nodes[l])
            D[:, j] += t
    return V, D


def _on(U, mats):
    """Applies a 1D matrix to each of the last three axes (z, y, x order); None leaves the axis."""
    for ax, M in zip((-1, -2, -3), mats):
        if M is not None:
            U = torch.matmul(U.movedim(ax, -1), M.T).movedim(-1, ax)
    return U


def _turns():
    """The 24 rotations of a cell: (axes, flips) with old coordinate a = new coordinate axes[a], reversed where flips[a]."""
    out = []
    for axes in ((0, 1, 2), (1, 2, 0), (2, 0, 1), (1, 0, 2), (0, 2, 1), (2, 1, 0)):
        even = axes in ((0, 1, 2), (1, 2, 0), (2, 0, 1))
        for f in range(8):
            flips = (f & 1, (f >> 1) & 1, f >> 2)
            if (sum(flips) % 2 == 0) == even:
                out.append((axes, flips))
    return out


def _old_of_new(U, turn):
    """U[..., z, y, x] in a turned cell's own coordinates -> in the box's."""
    axes, flips = turn
    lead = U.dim() - 3
    U = U.permute(*range(lead), *[lead + 2 - axes[a] for a in (2, 1, 0)])
    back = [lead + 2 - a for a in range(3) if flips[a]]
    return U.flip(back) if back else U


def _new_of_old(U, turn):
    axes, flips = turn
    lead = U.dim() - 3
    back = [lead + 2 - a for a in range(3) if flips[a]]
    U = U.flip(back) if back else U
    place = [0, 0, 0]
    for i, a in enumerate((2, 1, 0)):
        place[2 - axes[a]] = lead + i
    return U.permute(*range(lead), *place)


def _hex_mesh(m0, m1, m2):
    """A box of distorted hexahedra as a mesh generator would give it: vertices and cells in no order, each cell turned.
    Returns vertices, cells, the old cell of each new one and each new cell's turn (the last two and the box's vertices
    are what the plain reference needs)."""
    r = np.random.RandomState(7)
    g = (m0 + 1, m1 + 1, m2 + 1)
    Z, Y, X = np.meshgrid(*[np.arange(g[a]) for a in (2, 1, 0)], indexing="ij")
    ijk = [X.ravel(), Y.ravel(), Z.ravel()]
    V = np.stack([ijk[a] / (g[a] - 1) for a in range(3)], 1)
    inner = np.all([(ijk[a] > 0) & (ijk[a] < g[a] - 1) for a in range(3)], 0)
    for a in range(3):
        V[:, a] += np.where(inner, 0.2 / (g[a] - 1) * r.uniform(-1, 1, len(V)), 0)
    E = m0 * m1 * m2
    e = np.arange(E)
    i0, i1, i2 = e % m0, (e // m0) % m1, e // (m0 * m1)
    box = np.stack([(i0 + (v & 1)) + g[0] * ((i1 + ((v >> 1) & 1)) + g[1] * (i2 + (v >> 2))) for v in range(8)], 1)
    vnew, order, turn = r.permutation(len(V)), r.permutation(E), r.randint(0, 24, E)
    W = np.empty_like(V)
    W[vnew] = V
    ids = torch.from_numpy(vnew[box[order]]).view(E, 2, 2, 2)
    cells = torch.empty_like(ids)
    for t, tn in enumerate(_turns()):
        at = torch.from_numpy(np.nonzero(turn == t)[0])
        cells[at] = _new_of_old(ids[at], tn)
    return W, cells.reshape(E, 8).numpy().astype(np.int32), (order, turn), V[box]


class _Plain:
    """The SIPG operator and the FE operator on a box of cells, by dense 1D matrices in 64 bits; Dirichlet sides."""

    def __init__(self, m, k, nodes, device):
        """nodes: mapping nodes of each cell [cell][z][y][x][3], tensor GL points of any degree."""
        self.m, self.k, self.n = m, k, k + 1
        E, n = m[0] * m[1] * m[2], k + 1
        self.E, self.device = E, device
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=device)  # noqa: E731
        gl = _lobatto(n)
        xq, wq = np.polynomial.legendre.leggauss(n)
        xq, wq = (xq + 1) / 2, wq / 2
        S, D = _lagrange(gl, xq)
        ends, dends = _lagrange(gl, np.array([0.0, 1.0]))
        self.S, self.D, self.dend, self.w1 = t(S), t(D), t(dends), t(wq)
        mg = _lobatto(nodes.shape[1])
        mS, mD = (t(a) for a in _lagrange(mg, xq))
        mE, mdE = (t(a) for a in _lagrange(mg, np.array([0.0, 1.0])))
        X = [t(nodes[..., c]) for c in range(3)]

        def jacobian(val, der):   # val[a], der[a]: the 1D matrices of direction a
            return torch.stack([torch.stack([_on(X[c], [der[b] if b == a else val[b] for b in range(3)])
                                             for a in range(3)], -1) for c in range(3)], -2)
        w = self.w1
        J = jacobian([mS] * 3, [mD] * 3)
        Ji = torch.linalg.inv(J)
        wj = torch.linalg.det(J).abs() * (w[:, None, None] * w[None, :, None] * w[None, None, :])
        self.G = torch.einsum("ezyxac,ezyxbc->abezyx", Ji, Ji) * wj
        vol = wj.sum((1, 2, 3))
        del J, Ji
        # faces: [d][s] own area element and J^-1 n on [cell][t2][t1]
        self.dA, self.c, area = {}, {}, torch.zeros(E, dtype=torch.float64, device=device)
        ijk = self.ijk()
        for d in range(3):
            for s in range(2):
                Jf = jacobian([mE[s:s + 1] if a == d else mS for a in range(3)],
                              [mdE[s:s + 1] if a == d else mD for a in range(3)]).squeeze(3 - d)
                Ji = torch.linalg.inv(Jf)
                nv = Ji[..., d, :] * (1 if s else -1)
                length = nv.norm(dim=-1)
                self.dA[d, s] = torch.linalg.det(Jf).abs() * length * (w[:, None] * w[None, :])
                self.c[d, s] = torch.einsum("eqrac,eqrc->aeqr", Ji, nv / length[..., None])
                edge = ijk[d] == (m[d] - 1 if s else 0)
                area += self.dA[d, s].sum((1, 2)) * torch.where(edge, 1.0, 0.5)
        self.tau = n * n * area / vol

    def ijk(self):
        e = torch.arange(self.E, device=self.device)
        return e % self.m[0], (e // self.m[0]) % self.m[1], e // (self.m[0] * self.m[1])

    def other(self, a, d, s):
        """a[cell, ...] of the neighbour across face (d, s), NaN-free, and where there is none."""
        e = torch.arange(self.E, device=self.device)
        step = (1, self.m[0], self.m[0] * self.m[1])[d]
        edge = self.ijk()[d] == (self.m[d] - 1 if s else 0)
        return a[torch.where(edge, e, e + (step if s else -step))], edge

    def cells(self, U):
        """The cell term of U [cell][z][y][x]."""
        S, D = self.S, self.D
        g = [_on(U, [D if b == a else S for b in range(3)]) for a in range(3)]
        out = 0
        for a in range(3):
            f = sum(self.G[a, b] * g[b] for b in range(3))
            out = out + _on(f, [(D if b == a else S).T for b in range(3)])
        return out

    def face_mats(self, d, der=None):
        return [self.D if a == der else self.S for a in range(3) if a != d]

    @staticmethod
    def on_face(F, mats):
        """1D matrices on the last two axes of F [...][t2][t1]; mats = [of t1, of t2]."""
        return torch.matmul(torch.matmul(F, mats[0].T).transpose(-1, -2), mats[1].T).transpose(-1, -2)

    def apply(self, u):
        n = self.n
        U = u.reshape(self.E, n, n, n)
        out = self.cells(U)
        for d in range(3):
            tr = []
            others = [a for a in range(3) if a != d]
            for s in range(2):
                end = U.select(3 - d, n - 1 if s else 0)
                nd = torch.tensordot(U, self.dend[s], dims=([3 - d], [0]))
                g = {d: self.on_face(nd, self.face_mats(d))}
                for a in others:
                    g[a] = self.on_face(end, self.face_mats(d, a))
                c = self.c[d, s]
                tr.append((self.on_face(end, self.face_mats(d)), sum(c[a] * g[a] for a in range(3))))
            for s in range(2):
                v, q = tr[s]
                (vn, edge), (qn, _) = self.other(tr[1 - s][0], d, s), self.other(tr[1 - s][1], d, s)
                tn, _ = self.other(self.tau, d, s)
                at = edge[:, None, None]
                vn, qn = torch.where(at, -v, vn), torch.where(at, -q, qn)   # the mirror principle
                A = self.dA[d, s] * (torch.maximum(self.tau, tn)[:, None, None] * (v - vn) - (q - qn) / 2)
                B = -self.dA[d, s] * (v - vn) / 2
                c = self.c[d, s]
                end = self.on_face(A, [M.T for M in self.face_mats(d)])
                for a in others:
                    end = end + self.on_face(B * c[a], [M.T for M in self.face_mats(d, a)])
                out.select(3 - d, n - 1 if s else 0).add_(end)
                nd = self.on_face(B * c[d], [M.T for M in self.face_mats(d)])
                out += nd.unsqueeze(3 - d) * self.dend[s].reshape([-1 if ax == 3 - d else 1 for ax in range(4)])
        return out.reshape(-1)

    def cell_diagonal(self):
        S, D = self.S, self.D
        SS, DD, SD = (S * S).T, (D * D).T, (S * D).T
        out = 0
        for a in range(3):
            out = out + _on(self.G[a, a], [DD if b == a else SS for b in range(3)])
            for b in range(a):
                out = out + 2 * _on(self.G[a, b], [SD if e in (a, b) else SS for e in range(3)])
        return out

    def diagonal(self):
        n, S, D = self.n, self.S, self.D
        SS, SD = (S * S).T, (S * D).T
        out = self.cell_diagonal().contiguous()
        for d in range(3):
            others = [a for a in range(3) if a != d]
            for s in range(2):
                tn, edge = self.other(self.tau, d, s)
                twice = torch.where(edge, 2.0, 1.0)[:, None, None]
                dA, c = self.dA[d, s] * twice, self.c[d, s]
                f = self.on_face(dA * torch.maximum(self.tau, tn)[:, None, None], [SS, SS])
                f = f - self.on_face(dA * c[d], [SS, SS]) * self.dend[s, n - 1 if s else 0]
                for a in others:
                    f = f - self.on_face(dA * c[a], [SD if b == a else SS for b in others])
                out.select(3 - d, n - 1 if s else 0).add_(f)
        return out.reshape(-1)

    def fe(self):
        """(apply, diagonal, constrained) of the continuous space of the same degree."""
        n, k, m = self.n, self.k, self.m
        g = [m[a] * k + 1 for a in range(3)]
        c = self.ijk()
        i = torch.arange(n, device=self.device)
        at = [c[a][:, None] * k + i for a in range(3)]
        idx = (at[0][:, None, None, :] + g[0] * (at[1][:, None, :, None] + g[1] * at[2][:, :, None, None])).reshape(-1)
        p = torch.arange(g[0] * g[1] * g[2], device=self.device)
        q = (p % g[0], (p // g[0]) % g[1], p // (g[0] * g[1]))
        fixed = sum((q[a] == 0) | (q[a] == g[a] - 1) for a in range(3)) > 0
        free = (~fixed).to(torch.float64)

        def scatter(U):
            return torch.zeros(len(p), dtype=torch.float64, device=self.device).index_add_(0, idx, U.reshape(-1))

        def apply(u):
            v = scatter(self.cells((u * free)[idx].view(self.E, n, n, n)))
            return torch.where(fixed, u, v)
        return apply, torch.where(fixed, 1.0, scatter(self.cell_diagonal())), fixed

    def separable(self):
        """x -> P^-1 x with P the sum of three tensor products nearest to the operator of the undeformed box."""
        n, V, L = self.n, [], []
        S, D, w, de = self.S, self.D, self.w1, self.dend
        for d in range(3):
            h, md = 1.0 / self.m[d], self.m[d]
            K = torch.zeros(md * n, md * n, dtype=torch.float64, device=self.device)
            M = torch.zeros_like(K)
            tau = n * n * sum(self.m)
            e0, e1 = torch.eye(n, dtype=torch.float64, device=self.device)[[0, n - 1]]
            for i in range(md):
                at = slice(i * n, i * n + n)
                M[at, at] = h * S.T @ (w[:, None] * S)
                K[at, at] += D.T @ (w[:, None] * D) / h
            for f in range(md + 1):
                J, N = torch.zeros(2, md * n, dtype=torch.float64, device=self.device)
                both = 0.5 if 0 < f < md else 1.0
                if f > 0:
                    J[(f - 1) * n:f * n] += e1
                    N[(f - 1) * n:f * n] += both * de[1] / h
                if f < md:
                    J[f * n:f * n + n] -= e0
                    N[f * n:f * n + n] += both * de[0] / h
                K += -torch.outer(N, J) - torch.outer(J, N) + tau * (1 if both < 1 else 2) * torch.outer(J, J)
            R = self._half(M)
            lam, Q = torch.linalg.eigh(R @ K @ R)
            V.append(R @ Q)
            L.append(lam)
        lam = L[0][None, None, :] + L[1][None, :, None] + L[2][:, None, None]

        def solve(r):
            m = self.m
            lead = r.shape[:-1]
            R = r.view(*lead, m[2], m[1], m[0], n, n, n)
            o = len(lead)
            there = [*range(o), o, o + 3, o + 1, o + 4, o + 2, o + 5]
            R = R.permute(there).reshape(*lead, m[2] * n, m[1] * n, m[0] * n)
            R = _on(_on(R, [v.T for v in V]) / lam, V)
            R = R.view(*lead, m[2], n, m[1], n, m[0], n).permute(*range(o), o, o + 2, o + 4, o + 1, o + 3, o + 5)
            return R.reshape(r.shape)
        return solve

    @staticmethod
    def _half(M):
        """M^-1/2 of a block-diagonal mass matrix."""
        lam, Q = torch.linalg.eigh(M)
        return Q @ torch.diag(lam.rsqrt()) @ Q.T

    def solve(self, b):
        """A^-1 b by CG with the separable preconditioner; None if it takes too many steps."""
        pre = self.separable()
        x, r = torch.zeros_like(b), b.clone()
        z = pre(r)
        p, rz, stop = z.clone(), r @ z, 1e-13 * b.norm()
        for _ in range(600):
            Ap = self.apply(p)
            a = rz / (p @ Ap)
            x += a * p
            r -= a * Ap
            if r.norm() <= stop:
                return x
            z = pre(r)
            new = r @ z
            p = z + (new / rz) * p
            rz = new
        return None


def _box_nodes(m, deform):
    g = _lobatto(4 if deform else 2)
    ax = [(np.arange(m[a])[:, None] + g) / m[a] for a in range(3)]
    q = len(g)
    shape = (m[2], m[1], m[0], q, q, q)
    X = np.broadcast_to(ax[0][None, None, :, None, None, :], shape)
    Y = np.broadcast_to(ax[1][None, :, None, None, :, None], shape)
    Z = np.broadcast_to(ax[2][:, None, None, :, None, None], shape)
    P = np.stack([X, Y, Z], -1).reshape(-1, q, q, q, 3)
    if deform:
        P = P + 0.1 * np.prod(np.sin(np.pi * P), -1, keepdims=True)
    return P


def _eig_start(n):
    """The start vector of the eigenvalue estimate: SplitMix64 of 1910 xor i, uniform in [-1, 1)."""
    with np.errstate(over="ignore"):
        z = (np.arange(n, dtype=np.uint64) ^ np.uint64(1910)) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return 2 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1


def _largest(apply, dinv, r):
    """Largest eigenvalue of D^-1 A after 20 Jacobi-CG steps."""
    z = dinv * r
    p, rz, al, be = z.clone(), r @ z, [], []
    for _ in range(20):
        Ap = apply(p)
        a = rz / (p @ Ap)
        r = r - a * Ap
        z = dinv * r
        new = r @ z
        al.append(a.item())
        be.append((new / rz).item())
        p, rz = z + (new / rz) * p, new
    T = np.diag([1 / al[j] + (be[j - 1] / al[j - 1] if j else 0) for j in range(20)])
    for j in range(19):
        T[j, j + 1] = T[j + 1, j] = math.sqrt(be[j]) / al[j]
    return float(np.linalg.eigvalsh(T)[-1])


def _smooth(apply, diag, fixed, b, x):
    dinv = 1 / diag
    r0 = torch.as_tensor(_eig_start(len(b)), device=b.device)
    lam = _largest(apply, dinv, r0 if fixed is None else torch.where(fixed, 0.0, r0))
    hi, lo = 1.2 * lam, 0.06 * lam
    theta, delta = (hi + lo) / 2, (hi - lo) / 2
    old, rho = x, delta / theta
    x = x + dinv * (b - apply(x)) / theta
    for _ in range(1, STEPS):
        new = 1 / (2 * theta / delta - rho)
        x, old = x + new * rho * (x - old) + 2 * new / delta * dinv * (b - apply(x)), x
        rho = new
    return x


@lru_cache(maxsize=1)
def _plain(m, k, deform, device):
    return _Plain(m, k, _box_nodes(m, deform), device)


def exact(case, seed, device=None):
    device = device or ("cuda" if torch.cuda.is_available() else "cpu")
    kind, s = case["kind"], _inputs(case, seed, device)
    if kind == "batch":
        return [_plain((p["m"],) * 3, p["k"], 0, device).solve(b) for p, b in zip(_problems(case), s["b"])]
    m, k = _sizes(case), case["k"]
    if kind == "hex":
        _, _, (order, turn), corners = _hex_mesh(*m)
        P = _Plain(m, k, corners.reshape(-1, 2, 2, 2, 3), device)
        u = s["u"].double().view(-1, k + 1, k + 1, k + 1)
        U = torch.empty_like(u)
        which = [(torch.as_tensor(np.nonzero(turn == t)[0], device=device), tn) for t, tn in enumerate(_turns())]
        order = torch.as_tensor(order, device=device)
        for at, tn in which:
            U[order[at]] = _old_of_new(u[at], tn)
        V, v = P.apply(U).view_as(U), torch.empty_like(u)
        for at, tn in which:
            v[at] = _new_of_old(V[order[at]], tn)
        return v.reshape(-1)
    P = _plain(m, k, case["deform"], device)
    if kind == "apply":
        return P.apply(s["u"].double())
    if kind == "smooth":
        if case["level"] == "dg":
            return _smooth(P.apply, P.diagonal(), None, s["b"].double(), s["x0"].double())
        apply, diag, fixed = P.fe()
        return _smooth(apply, diag, fixed, s["b"].double(), s["x0"].double())
    if kind == "solve":
        return P.solve(s["b"])
    rows = [P.solve(b) for b in s["b"]]
    return None if any(x is None for x in rows) else torch.stack(rows)
