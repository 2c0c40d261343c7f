"""Cases by which the speed of the library is measured: the calls that a program
makes once per Newton step, over the sizes of the repository's own scenes.

A case names a call ("kind"), a scene and the options that the caller picks.
Scenes are drawn on the GPU from the case's seed with the recipes of the test
scenes: tet cubes of n^3 vertices (5 tets per cell, jittered rest positions, a
deformed state, lumped mass, contact pairs k n n^T with k log-uniform in
[1e2, 1e6], triplets in shuffled order as a parallel element loop emits them),
square cloth sheets, and affine cubes resting on a tet cube.  Tet stiffness is
linear elasticity on the deformed shape, which has the pattern and the spread
of values of the elastic Hessian.

Iterative calls run a fixed budget of iterations (a simulator's time-bounded
inexact Newton step: an unconverged solve still gives a descent direction), so
that every pass does the same work; "solve" and "grad" run to convergence.
With a low-precision preconditioner the iterates carry its own rounding (1e-7
and more), so those forms appear in solves to ten digits and in single applies.
The FP32-inner solve (gs_pcg_solve_mixed) is not among the cases: it is the
slowest of the precision forms on every scene the repository measures.
"""

import math

import numpy as np
import torch

from paper_2411_06224_gb300 import autograd as G
from paper_2411_06224_gb300 import binding as B

DEV = "cuda"
F64 = torch.float64
PREC = {"fp64": B.GS_PREC_FP64, "fp32": B.GS_PREC_FP32, "bf16": B.GS_PREC_BF16}
SPMV = {"row": B.GS_SPMV_ROW, "ff": B.GS_SPMV_ROW_FF}
NU, RHO, DT = 0.4, 1000.0, 0.01
SHEET = dict(E=1e8, lam=0.05e6, thickness=1e-3, rho=200.0, dt=DT)


def listed():
    return [
        # one small body re-assembled every Newton step: launches and readbacks count
        dict(name="assemble tet16", kind="assemble", n=16, contacts=2000, near=False, E=1e5),
        # the assembly of the benchmark's system (13.4M triplets)
        dict(name="assemble tet64", kind="assemble", n=64, contacts=200_000, near=True, E=1e7),
        # a deformable body in contact with many affine bodies (two-level reduction)
        dict(name="assemble abd40", kind="abd", n=40, bodies=1000, contacts=100_000, E=1e6),
        # a new preconditioner for new values, then its first apply (default precision)
        dict(name="build tet64 fp64", kind="build", n=64, contacts=200_000, near=True, E=1e7, N=32, L=3, prec="fp64",
             nrhs=1),
        # the benchmark's smallest form, whole: assembly, build and solve to 1e-6
        dict(name="solve tet16", kind="solve", n=16, contacts=2000, near=False, E=1e5, N=32, L=2, prec="fp64", nrhs=4,
             spmv="ff", tol=1e-6),
        # the benchmark's PCG: many right-hand sides on the large body
        dict(name="pcg tet64 fp64 rhs8", kind="pcg", scene="tet", n=64, contacts=200_000, near=True, E=1e7, N=32, L=3,
             prec="fp64", nrhs=8, spmv="ff", iters=24),
        # one right-hand side with the binding's default options, an odd size
        dict(name="pcg tet45 fp64 rhs1", kind="pcg", scene="tet", n=45, contacts=70_000, near=True, E=1e6, N=32, L=3,
             prec="fp64", nrhs=1, spmv="row", iters=24),
        # the FP32 preconditioner, to ten digits (as differentiation asks): assembly, build, many iterations
        dict(name="solve tet40 fp32", kind="solve", n=40, contacts=10_000, near=True, E=1e5, N=32, L=3, prec="fp32",
             nrhs=4, spmv="ff", tol=1e-10),
        # many uneven bodies solved together in one graph
        dict(name="batch 24 bodies", kind="batch", systems=24, vmin=1000, vmax=30_000, E=1e6, N=32, L=3, prec="fp64",
             iters=24),
        # forward and backward of a differentiable solve
        dict(name="grad tet20", kind="grad", n=20, contacts=400, near=True, E=1e5, N=32, L=3, prec="fp64", nrhs=2),
        # an implicit step of five Newton steps: element Hessians, numeric assembly, refresh, PCG, line search
        dict(name="newton tet32", kind="newton", n=32, springs=10_000, E=1e5, steps=5, N=32, L=3, prec="fp64", spmv="ff"),
        # element Hessians of a large sheet
        dict(name="cloth triplets 512", kind="cloth", n=512),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["assemble", "abd", "build", "solve", "pcg", "pcg", "batch", "grad", "newton", "cloth"])
    E = math.exp(rng.uniform(math.log(1e5), math.log(1e8)))
    mas = dict(N=rng.choice([32, 32, 16, 24]), L=rng.randint(2, 3), prec=rng.choice(["fp64", "fp64", "fp32", "bf16"]))
    tet = lambda lo, hi: (lambda n: dict(n=n, contacts=max(1, int(n ** 3 * rng.uniform(0.02, 0.8))),
                                         near=rng.random() < 0.7, E=E))(_logint(rng, lo, hi))
    if kind == "assemble":
        return dict(kind=kind, **tet(8, 64))
    if kind == "abd":
        return dict(kind=kind, n=_logint(rng, 12, 40), bodies=_logint(rng, 16, 1000),
                    contacts=_logint(rng, 500, 100_000), E=E)
    if kind == "build":
        return dict(kind=kind, nrhs=rng.randint(1, 8), **tet(10, 62), **mas)
    if kind == "solve":
        return dict(kind=kind, nrhs=rng.randint(1, 6), spmv=rng.choice(["row", "ff"]), **dict(tet(8, 24), E=1e5),
                    **mas, tol=1e-6 if mas["prec"] == "fp64" else 1e-10)
    if kind == "pcg":
        opts = dict(nrhs=rng.randint(1, 8), spmv=rng.choice(["row", "ff", "ff"]), iters=rng.randint(12, 24),
                    **dict(mas, prec="fp64"))
        if rng.random() < 0.3:
            return dict(kind=kind, scene="cloth", **dict(tet(40, 400), E=1e8, contacts=0), **opts)
        return dict(kind=kind, scene="tet", **tet(10, 62), **opts)
    if kind == "batch":
        return dict(kind=kind, systems=rng.randint(3, 24), vmin=500, vmax=_logint(rng, 2000, 30_000), E=E, iters=24,
                    **dict(mas, prec="fp64"))
    if kind == "grad":
        return dict(kind=kind, nrhs=rng.randint(1, 4), **dict(tet(8, 20), E=1e5), **dict(mas, prec="fp64"))
    if kind == "newton":
        n = _logint(rng, 8, 32)
        return dict(kind=kind, n=n, springs=_logint(rng, 10, n ** 3 // 3), E=1e5, steps=rng.randint(1, 5), spmv=rng.choice(["row", "ff"]),
                    **dict(mas, prec="fp64"))
    return dict(kind=kind, n=_logint(rng, 24, 500))


# ---------------------------------------------------------------- scenes
_SPLIT = (((1, 2, 4, 7), (0, 1, 2, 4), (3, 1, 7, 2), (5, 1, 4, 7), (6, 2, 7, 4)),
          ((0, 3, 5, 6), (1, 0, 5, 3), (2, 0, 3, 6), (4, 0, 6, 5), (7, 3, 6, 5)))
_PAIRS4 = [(a, b) for a in range(4) for b in range(a, 4)]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(shape, g):
    return torch.randn(shape, dtype=F64, device=DEV, generator=g)


def _rand(shape, g):
    return torch.rand(shape, dtype=F64, device=DEV, generator=g)


def _randint(hi, count, g, lo=0):
    return torch.randint(lo, hi, (count,), device=DEV, generator=g)


def _i32(t):
    return t.to(torch.int32).contiguous()


def _cube(n, g):
    """Rest positions, deformed positions and tets (positive volume) of the n^3 cube; vertex i + n j + n^2 k."""
    h = 1.0 / (n - 1)
    v = torch.arange(n ** 3, device=DEV)
    X = torch.stack([v % n, v // n % n, v // (n * n)], 1).to(F64) * h + _randn((n ** 3, 3), g) * (0.05 * h)
    c = torch.arange((n - 1) ** 3, device=DEV)
    ci, cj, ck = c % (n - 1), c // (n - 1) % (n - 1), c // (n - 1) ** 2
    o = torch.arange(8, device=DEV)
    corner = ((ci[:, None] + (o & 1)) + n * (cj[:, None] + (o >> 1 & 1)) + n * n * (ck[:, None] + (o >> 2 & 1)))
    odd = ((ci + cj + ck) & 1).bool()
    t0, t1 = (corner[:, torch.tensor(s, device=DEV)] for s in _SPLIT)
    tets = torch.where(odd[:, None, None], t1, t0).reshape(-1, 4)
    d = X[tets[:, 1:]] - X[tets[:, :1]]
    neg = (d[:, 0] * torch.linalg.cross(d[:, 1], d[:, 2], dim=1)).sum(1) < 0
    tets = torch.where(neg[:, None], tets[:, [0, 2, 1, 3]], tets)
    A = torch.eye(3, dtype=F64, device=DEV) + 0.2 * _rand((3, 3), g) - 0.1
    return X, X @ A.T + _randn((n ** 3, 3), g) * (0.02 * h), tets


def _weights(X, tets):
    """Volumes (T,) and shape gradients w (T, 4, 3)."""
    d = X[tets[:, 1:]] - X[tets[:, :1]]
    c = torch.stack([torch.linalg.cross(d[:, 1], d[:, 2], dim=1), torch.linalg.cross(d[:, 2], d[:, 0], dim=1),
                     torch.linalg.cross(d[:, 0], d[:, 1], dim=1)], 1)
    det = (d[:, 0] * c[:, 0]).sum(1)
    w = c / det[:, None, None]
    return det.abs() / 6.0, torch.cat([-w.sum(1, keepdim=True), w], 1)


def _distinct(i, j, V, count, g):
    """count distinct pairs (min, max) of the given ones, in random order."""
    key = torch.unique(torch.minimum(i, j) * V + torch.maximum(i, j))
    key = key[torch.randperm(key.numel(), device=DEV, generator=g)[:count]]
    return torch.stack([key // V, key % V], 1)


def _contact_pairs(n, count, near, g):
    """Near: half on mesh edges (they repeat), half distinct cell diagonals.  Else distinct pairs that are no neighbours.
    The number of distinct keys is that of the case, whatever the seed."""
    V = n ** 3
    if not near:
        i, j = _randint(V, 3 * count + 64, g), _randint(V, 3 * count + 64, g)
        far = (i % n - j % n).abs() > 1
        return _distinct(i[far], j[far], V, count, g)
    edge = count - count // 2
    ax, i = _randint(3, edge, g), _randint(V, edge, g)
    q = torch.stack([i % n, i // n % n, i // (n * n)], 1)
    q.scatter_(1, ax[:, None], q.gather(1, ax[:, None]).clamp(max=n - 2))
    i = q[:, 0] + n * q[:, 1] + n * n * q[:, 2]
    edges = torch.stack([i, i + torch.tensor([1, n, n * n], device=DEV)[ax]], 1)
    c = torch.randperm((n - 1) ** 3 * 4, device=DEV, generator=g)[: count // 2]  # cell and diagonal
    d, c = c % 4, c // 4
    o = torch.stack([c % (n - 1), c // (n - 1) % (n - 1), c // (n - 1) ** 2], 1)
    flip = torch.stack([torch.zeros_like(d), d & 1, d >> 1], 1)
    at = lambda t: t[:, 0] + n * t[:, 1] + n * n * t[:, 2]
    u, v = at(o + flip), at(o + 1 - flip)
    return torch.cat([edges, torch.stack([torch.minimum(u, v), torch.maximum(u, v)], 1)])


def _springs_k(count, lo, hi, g):
    nv = _randn((count, 3), g)
    nv = nv / nv.norm(dim=1, keepdim=True)
    k = torch.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * _rand((count,), g))
    return k[:, None, None] * nv[:, :, None] * nv[:, None, :]


def _tet_triplets(x, tets, E):
    """Element stiffness (10 upper blocks per tet) and lumped mass blocks."""
    vol, w = _weights(x, tets)
    mu, lam = E / (2 * (1 + NU)), E * NU / ((1 + NU) * (1 - 2 * NU))
    pa, pb = (torch.tensor(p, device=DEV) for p in zip(*_PAIRS4))
    wa, wb = w[:, pa], w[:, pb]
    blk = lam * wa[..., :, None] * wb[..., None, :] + mu * wb[..., :, None] * wa[..., None, :]
    blk += (mu * (wa * wb).sum(-1))[..., None, None] * torch.eye(3, dtype=F64, device=DEV)
    blk *= vol[:, None, None, None]
    r, c = tets[:, pa], tets[:, pb]
    blk = torch.where((r > c)[..., None, None], blk.transpose(-1, -2), blk)
    m = torch.zeros(x.shape[0], dtype=F64, device=DEV)
    m.index_put_((tets.reshape(-1),), (RHO / DT ** 2 / 4 * vol).repeat_interleave(4), accumulate=True)
    v = torch.arange(x.shape[0], device=DEV)
    return (torch.cat([torch.minimum(r, c).reshape(-1), v]), torch.cat([torch.maximum(r, c).reshape(-1), v]),
            torch.cat([blk.reshape(-1, 3, 3), m[:, None, None] * torch.eye(3, dtype=F64, device=DEV)]))


def _contact_triplets(pairs, K):
    i, j = pairs[:, 0], pairs[:, 1]
    return torch.cat([i, j, i]), torch.cat([i, j, j]), torch.cat([K, K, -K])


def _edges(elements):
    """Distinct undirected vertex pairs of elements (E, 2)."""
    k = elements.shape[1]
    p = torch.cat([elements[:, [a, b]] for a in range(k) for b in range(a + 1, k)]).sort(1).values
    V = int(elements.max()) + 1
    key = torch.unique(p[:, 0] * V + p[:, 1])
    return torch.stack([key // V, key % V], 1)


def _csr(V, edges):
    key = torch.cat([edges[:, 0] * V + edges[:, 1], edges[:, 1] * V + edges[:, 0]]).sort().values
    ptr = torch.searchsorted(key, torch.arange(V + 1, device=DEV) * V)
    return _i32(ptr), _i32(key % V)


class _Scene:
    """Triplets, rest positions and graph of one system."""

    def __init__(self, V, X, trip, edges, contacts, g):
        perm = torch.randperm(trip[0].numel(), device=DEV, generator=g)
        self.V, self.X, self.edges, self.contacts = V, X.contiguous(), edges, contacts
        self.rows, self.cols, self.blocks = _i32(trip[0][perm]), _i32(trip[1][perm]), trip[2][perm].contiguous()


def _tet_scene(case, seed):
    g = _gen(seed)
    n = case["n"]
    X, x, tets = _cube(n, g)
    pairs = _contact_pairs(n, case["contacts"], case["near"], g)
    t, c = _tet_triplets(x, tets, case["E"]), _contact_triplets(pairs, _springs_k(pairs.shape[0], 1e2, 1e6, g))
    return _Scene(n ** 3, X, [torch.cat(p) for p in zip(t, c)], _edges(tets), pairs, g), g


def _sheet(n, g):
    """Rest and deformed positions, triangles and hinges of an n x n sheet (2 % stretched, sheared, rippled)."""
    h = 1.0 / (n - 1)
    v = torch.arange(n * n, device=DEV)
    X = torch.stack([v % n * h, v // n * h, torch.zeros(n * n, dtype=F64, device=DEV)], 1).to(F64)
    A = torch.eye(3, dtype=F64, device=DEV)
    A[0, 0], A[0, 1] = 1.02, 0.1 * float(_rand((1,), g))
    x = X @ A.T + _randn(X.shape, g) * (0.01 * h)
    q = torch.arange((n - 1) ** 2, device=DEV)
    a = q % (n - 1) + n * (q // (n - 1))
    tris = torch.cat([torch.stack([a, a + 1, a + n + 1], 1), torch.stack([a, a + n + 1, a + n], 1)])
    e = torch.cat([tris[:, [0, 1]], tris[:, [1, 2]], tris[:, [2, 0]]])
    opp = torch.cat([tris[:, 2], tris[:, 0], tris[:, 1]])
    key, order = torch.sort(e.min(1).values * (n * n) + e.max(1).values, stable=True)
    i0 = torch.nonzero(key[1:] == key[:-1]).reshape(-1)
    i0, i1 = order[i0], order[i0 + 1]
    return X, x, tris, torch.stack([e[i0, 0], e[i0, 1], opp[i0], opp[i1]], 1)


def _cloth_scene(case, seed):
    g = _gen(seed)
    X, x, tris, hinges = _sheet(case["n"], g)
    r, c, b = _cloth_blocks(X, x, tris, hinges)
    edges = torch.unique(torch.cat([_edges(hinges), _edges(tris)]), dim=0)
    return _Scene(X.shape[0], X, (r, c, b), edges, torch.zeros((0, 2), dtype=torch.int64, device=DEV), g), g


def _abd_scene(case, seed):
    """A tet cube with 2 cm affine cubes on a grid over its top face; contacts body-vertex, body-body, vertex-vertex."""
    g = _gen(seed)
    n, nb, P = case["n"], case["bodies"], case["contacts"]
    V, size = n ** 3, 0.02
    X, x, tets = _cube(n, g)
    rows, cols, blocks = (list(p) for p in zip(_tet_triplets(x, tets, case["E"])))
    n_nodes = V + 8 * nb
    corner = torch.stack([torch.arange(8, device=DEV) >> s & 1 for s in range(3)], 1).to(F64) * size - size / 2
    node = torch.arange(V, n_nodes, device=DEV)
    eye = torch.eye(3, dtype=F64, device=DEV)
    rows.append(node), cols.append(node), blocks.append((RHO * size ** 3 / 8 / DT ** 2 * eye).expand(8 * nb, 3, 3))
    # orthogonality potential on the bodies' own rows a_1..a_3: 4 kv (delta_kl sum a a^T + a_l a_k^T)
    A = eye + 0.01 * _randn((nb, 3, 3), g)
    S = A @ A.transpose(1, 2)
    for k in range(3):
        for l in range(k, 3):
            H = A[:, :, l, None] * A[:, :, k][:, None, :] + (S if k == l else 0.0)
            own = n_nodes + 4 * torch.arange(nb, device=DEV)
            rows.append(own + 1 + k), cols.append(own + 1 + l), blocks.append(4e11 * size ** 3 * H)
    a, b = P // 2, P // 4
    # a body corner and one of the four top-face vertices nearest below it (each once, then again at random); a
    # corner and one of the next body
    grid = math.ceil(math.sqrt(nb))
    pick = torch.arange(a, device=DEV)
    pick = torch.where(pick < 32 * nb, pick, _randint(32 * nb, a, g))
    ca = pick // 4
    centre = torch.stack([ca // 8 % grid, ca // 8 // grid], 1).to(F64)
    cell = (((centre + 0.5) / grid + corner[ca % 8, :2]) * (n - 1)).floor().long().clamp(0, n - 2)
    top = cell[:, 0] + (pick & 1) + n * (cell[:, 1] + (pick >> 1 & 1)) + n * n * (n - 1)
    first = torch.arange(b, device=DEV) % (nb - 1)
    c0, c1 = V + 8 * first + _randint(8, b, g), V + 8 * (first + 1) + _randint(8, b, g)
    pairs = torch.cat([torch.stack([top, V + ca], 1), torch.stack([c0, c1], 1),
                       _contact_pairs(n, P - a - b, True, g)])
    for part, q in zip((rows, cols, blocks), _contact_triplets(pairs, _springs_k(pairs.shape[0], 1e2, 1e6, g))):
        part.append(q)
    sc = _Scene(V, X, [torch.cat(p) for p in (rows, cols, blocks)], None, pairs, g)
    sc.n_nodes = n_nodes
    sc.body = _i32(torch.cat([torch.full((V,), -1, device=DEV), (node - V) // 8]))
    sc.xbar = torch.cat([torch.zeros((V, 3), dtype=F64, device=DEV), corner.repeat(nb, 1)]).contiguous()
    return sc


def _batch_scene(case, seed):
    """Cubes of uneven size spread over [vmin, vmax] vertices, and of three stiffnesses."""
    S, out, sizes = case["systems"], [], []
    for s in range(S):
        V = case["vmin"] * (case["vmax"] / case["vmin"]) ** (s / max(S - 1, 1))
        n = max(3, round(V ** (1 / 3)))
        E = case["E"] * 10.0 ** (s % 3 - 1)
        sc, g = _tet_scene(dict(n=n, contacts=max(1, n ** 3 // 20), near=False, E=E), seed * 1000 + s)
        out.append(sc), sizes.append(sc.V)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    shift = lambda f: torch.cat([f(s) + int(o) for s, o in zip(out, off)])
    sc = out[0]
    sc.rows, sc.cols = _i32(shift(lambda s: s.rows)), _i32(shift(lambda s: s.cols))
    sc.edges, sc.contacts = shift(lambda s: s.edges), shift(lambda s: s.contacts)
    sc.blocks, sc.X = torch.cat([s.blocks for s in out]), torch.cat([s.X for s in out])
    sc.V = int(off[-1])
    return sc, off, g


def _elastic_scene(case, seed):
    g = _gen(seed)
    n = case["n"]
    X, x, tets = _cube(n, g)
    om = _randn((3,), g)
    om *= 10.0 / om.norm()  # rad/s
    xt = x + DT * torch.linalg.cross(om.expand_as(x), x - x.mean(0), dim=1)
    pairs = _contact_pairs(n, case["springs"], False, g)
    return X, x.contiguous(), xt.contiguous(), tets, pairs, _springs_k(pairs.shape[0], 1e2, 1e4, g).contiguous()


# ---------------------------------------------------------------- calls
_CTX = None


def _ctx():
    global _CTX
    if _CTX is None:  # a program keeps one context
        _CTX = B.gs_create(0)
    return _CTX


class _State:
    """Tensors and handles that a program holds before the call."""

    def __init__(self, case):
        self.case, self.kind, self.freed = case, case["kind"], []

    def own(self, handle, destroy):
        self.freed.append((handle, destroy))
        return handle

    def __del__(self):
        try:
            for h, destroy in reversed(self.freed):
                destroy(h)
        except Exception:  # noqa: BLE001 - interpreter shutdown
            pass


def _graph(st, sc):
    st.X, st.V = sc.X, sc.V
    st.adj_ptr, st.adj = _csr(sc.V, sc.edges)
    st.contacts = _i32(sc.contacts) if sc.contacts.shape[0] else None


def _trip(st, sc):
    st.V, st.rows, st.cols, st.blocks = sc.V, sc.rows, sc.cols, sc.blocks


def _build(st, mat, **kw):
    c = st.case
    return B.gs_build_mas_mesh(_ctx(), mat, st.X, st.adj_ptr, st.adj, st.contacts, domain_size=c["N"],
                               max_levels=c["L"], precision=PREC[c["prec"]], **kw)


def prepare(case, seed):
    st = _State(case)
    ctx = _ctx()
    kind = st.kind
    if kind == "assemble":
        _trip(st, _tet_scene(case, seed)[0])
    elif kind == "abd":
        sc = _abd_scene(case, seed)
        _trip(st, sc)
        st.n_nodes, st.body, st.xbar = sc.n_nodes, sc.body, sc.xbar
    elif kind in ("build", "pcg", "solve"):
        sc, g = (_cloth_scene if case.get("scene") == "cloth" else _tet_scene)(case, seed)
        _graph(st, sc)
        st.b = _randn((case["nrhs"], 3 * sc.V), g)
        if kind == "solve":
            _trip(st, sc)
        else:
            st.mat = st.own(B.gs_assemble(ctx, sc.V, sc.rows, sc.cols, sc.blocks), B.gs_mat_destroy)
        if kind == "pcg":
            st.mas = st.own(_build(st, st.mat), B.gs_mas_destroy)
    elif kind == "batch":
        sc, st.off, g = _batch_scene(case, seed)
        st.b = _randn((3 * sc.V,), g)
        adj_ptr, adj = _csr(sc.V, sc.edges)
        mp, nd = B.gs_partition_batch(sc.X.cpu().numpy(), st.off, case["N"])
        st.mat = st.own(B.gs_assemble(ctx, sc.V, sc.rows, sc.cols, sc.blocks), B.gs_mat_destroy)
        st.mas = st.own(B.gs_build_mas(ctx, st.mat, torch.as_tensor(mp, device=DEV), nd, adj_ptr, adj,
                                       _i32(sc.contacts), domain_size=case["N"], max_levels=case["L"],
                                       precision=PREC[case["prec"]]), B.gs_mas_destroy)
    elif kind == "grad":
        sc, g = _tet_scene(case, seed)
        h = lambda t: t.cpu().numpy()
        ptr, adj = _csr(sc.V, sc.edges)
        st.system = G.System(ctx, sc.V, h(sc.rows), h(sc.cols), h(sc.X), h(ptr), h(adj), h(sc.contacts),
                             domain_size=case["N"], max_levels=case["L"], precision=PREC[case["prec"]])
        st.blocks = sc.blocks.requires_grad_(True)
        st.b = _randn((case["nrhs"], 3 * sc.V), g).requires_grad_(True)
        st.gx = _randn((case["nrhs"], 3 * sc.V), g)
    elif kind == "newton":
        X, st.x0, st.xt, tets, pairs, K = _elastic_scene(case, seed)
        st.adj_ptr, st.adj = _csr(X.shape[0], _edges(tets))
        st.fem = st.own(B.gs_fem_create(ctx, X.contiguous(), _i32(tets), case["E"], NU, RHO, DT), B.gs_fem_destroy)
        B.gs_fem_set_springs(ctx, st.fem, _i32(pairs), K, (X[pairs[:, 0]] - X[pairs[:, 1]]).contiguous())
    else:
        X, x, tris, hinges = _sheet(case["n"], _gen(seed))
        st.x = x.contiguous()
        st.cloth = st.own(B.gs_cloth_create(ctx, X.contiguous(), _i32(tris), _i32(hinges), **SHEET), B.gs_cloth_destroy)
    return st


def run(st):
    ctx, case, kind = _ctx(), st.case, st.kind
    if kind == "assemble" or kind == "abd":
        if kind == "abd":
            m = B.gs_assemble_abd(ctx, st.n_nodes, st.V, case["bodies"], st.body, st.xbar, st.rows, st.cols, st.blocks)
        else:
            m = B.gs_assemble(ctx, st.V, st.rows, st.cols, st.blocks)
        out = B.gs_mat_export(ctx, m)
        B.gs_mat_destroy(m)
        return out
    if kind == "build":
        mas = _build(st, st.mat)
        z = torch.empty_like(st.b)
        B.gs_mas_apply(ctx, mas, st.b, z, nrhs=case["nrhs"])
        B.gs_mas_destroy(mas)
        return z
    if kind == "solve":
        mat = B.gs_assemble(ctx, st.V, st.rows, st.cols, st.blocks)
        mas = _build(st, mat)
        x = torch.empty_like(st.b)
        B.gs_pcg_solve(ctx, mat, mas, st.b, x, nrhs=case["nrhs"], tol=case["tol"], variant=SPMV[case["spmv"]])
        B.gs_mas_destroy(mas)
        B.gs_mat_destroy(mat)
        return x
    if kind == "pcg":
        x = torch.empty_like(st.b)
        _, rel, _ = B.gs_pcg_solve(ctx, st.mat, st.mas, st.b, x, nrhs=case["nrhs"], tol=1e-8, max_iter=case["iters"],
                                   variant=SPMV[case["spmv"]], raise_on_maxiter=False)
        return x, rel
    if kind == "batch":
        x = torch.empty_like(st.b)
        _, rel, _ = B.gs_pcg_solve_batch(ctx, st.mat, st.mas, st.off, st.b, x, tol=1e-8, max_iter=case["iters"],
                                         raise_on_maxiter=False)
        return x, rel
    if kind == "grad":
        x = G.solve(st.blocks, st.b, st.system)
        db, dblocks = torch.autograd.grad(x, (st.b, st.blocks), st.gx)
        return x.detach(), db, dblocks
    if kind == "newton":
        x = st.x0.clone()
        _, energies, _ = B.gs_fem_newton(ctx, st.fem, st.xt, x, st.adj_ptr, st.adj, spmv_variant=SPMV[case["spmv"]],
                                             domain_size=case["N"], max_levels=case["L"], precision=PREC[case["prec"]],
                                         tol=0.0, max_newton=case["steps"], raise_on_maxiter=False)
        return x, energies[-1]
    return B.gs_cloth_triplets(ctx, st.cloth, st.x)


# ---------------------------------------------------------------- work
def _stored(n):
    """Stored blocks of the n^3 cube: vertices, grid edges and one diagonal per cell face."""
    return n ** 3 + 3 * n * n * (n - 1) + 3 * n * (n - 1) ** 2


def _solver_bytes(n, U, N, nrhs):
    """(matrix, symmetric domain inverses, one vector) in bytes."""
    ld = 3 * N
    return 76 * U, -(-n // N) * ld * (ld + 1) / 2 * 8, 24 * n * nrhs


def _pcg_work(n, U, case, nrhs, iters):
    a, m, v = _solver_bytes(n, U, case["N"], nrhs)
    m *= {"fp64": 1.0, "fp32": 0.5, "bf16": 0.25}[case["prec"]]
    # per iteration the matrix and the inverses once, x, r and p read and written, Ap and z written and read
    return dict(bytes=iters * (a + m + 10 * v), flops=iters * nrhs * (18 * (2 * U - n) + 6 * 3 * case["N"] * n + 36 * n))


def work(case):
    kind, n = case["kind"], case.get("n", 0)
    if kind == "cloth":
        T, H, V = 2 * (n - 1) ** 2, 3 * (n - 1) ** 2 - 2 * (n - 1), n * n
        K = 6 * T + 10 * H + V
        return dict(bytes=80 * K + 68 * T + 24 * H + 32 * V, flops=300 * T + 181 * H)
    V, T = n ** 3, 5 * (n - 1) ** 3
    if kind == "batch":
        S = case["systems"]
        sizes = [max(3, round((case["vmin"] * (case["vmax"] / case["vmin"]) ** (s / max(S - 1, 1))) ** (1 / 3)))
                 for s in range(S)]
        V, U = sum(q ** 3 for q in sizes), sum(_stored(q) + q ** 3 // 20 for q in sizes)
        return _pcg_work(V, U, case, 1, case["iters"])
    if case.get("scene") == "cloth":
        V = n * n
        U = V + 2 * n * (n - 1) + (n - 1) ** 2 + 3 * (n - 1) ** 2
        return _pcg_work(V, U, case, case["nrhs"], case["iters"])
    if kind == "newton":
        U = _stored(n) + case["springs"]
        a, m, v = _solver_bytes(V, U, case["N"], 1)
        steps, it = case["steps"], 35  # PCG iterations of a Newton step, as these scenes take
        return dict(bytes=steps * (936 * T + 72 * (10 * T + U) + 3 * m + it * (a + m + 10 * v)),
                    flops=steps * (3300 * T + (3 * case["N"]) ** 2 * 3 * V))
    K = 10 * T + V + 3 * case["contacts"]
    U = _stored(n) + case["contacts"] // (2 if case.get("near", True) else 1)
    if kind == "abd":
        nb, P = case["bodies"], case["contacts"]
        K += 8 * nb + 6 * nb
        U += 4 * min(P // 2, 12 * nb) + 26 * nb
    asm = dict(bytes=80 * (K + U), flops=9 * K)
    if kind in ("assemble", "abd"):
        return asm
    if kind == "pcg":
        return _pcg_work(V, U, case, case["nrhs"], case["iters"])
    a, m, v = _solver_bytes(V, U, case["N"], case["nrhs"])
    build = dict(bytes=a + 2 * m + 2 * v, flops=(3 * case["N"]) ** 2 * 3 * V)  # Cholesky, its inverse, their product
    if kind == "build":
        return build
    pcg = _pcg_work(V, U, case, case["nrhs"], 100 if case.get("tol") == 1e-6 else 300)
    return {k: asm[k] + build[k] + pcg[k] for k in asm}


# ---------------------------------------------------------------- 64-bit values
def _sum_blocks(n, r, c, b):
    key, inv = torch.unique(r.long() * n + c.long(), return_inverse=True)
    au = torch.zeros((key.numel(), 9), dtype=F64, device=DEV).index_add_(0, inv, b.reshape(-1, 9))
    return _i32(key // n), _i32(key % n), au.reshape(-1, 3, 3)


class _Matrix:
    def __init__(self, n, r, c, b):
        self.n = n
        rid, cid, self.au = _sum_blocks(n, r, c, b)
        self.rid, self.cid = rid.long(), cid.long()
        self.off = self.rid != self.cid

    def __call__(self, x):  # (n, 3, k)
        o = self.off
        y = torch.zeros_like(x).index_add_(0, self.rid, self.au @ x[self.cid])
        return y.index_add_(0, self.cid[o], self.au[o].transpose(1, 2) @ x[self.rid[o]])


def _bisection(X, N):
    """Slots of the recursive coordinate bisection: widest axis, order by (coordinate, index), N ceil(P / 2) left."""
    n = X.shape[0]
    part = torch.zeros(n, dtype=torch.int64, device=DEV)
    node = torch.arange(n, device=DEV)
    while True:
        size = torch.bincount(part)
        P = -(-size // N)
        if int(P.max()) <= 1:
            return N * part + _rank(part, node)
        S = size.numel()
        at = part[:, None].expand(-1, 3)
        lo = torch.full((S, 3), math.inf, dtype=F64, device=DEV).scatter_reduce_(0, at, X, "amin")
        ext = torch.full((S, 3), -math.inf, dtype=F64, device=DEV).scatter_reduce_(0, at, X, "amax") - lo
        axis = torch.where((ext[:, 1] > ext[:, 0]) & (ext[:, 1] >= ext[:, 2]), 1, 0)
        axis = torch.where((ext[:, 2] > ext[:, 0]) & (ext[:, 2] > ext[:, 1]), 2, axis)
        order = torch.argsort(X[node, axis[part]], stable=True)
        left = torch.where(P > 1, N * ((P + 1) // 2), size)
        right = _rank(part, order) >= left[part]
        part = torch.unique(2 * part + right, return_inverse=True)[1]


def _rank(part, order):
    """Rank of every node within its part along `order`."""
    order = order[torch.argsort(part[order], stable=True)]
    start = torch.cumsum(torch.bincount(part), 0) - torch.bincount(part)
    rank = torch.empty_like(part)
    rank[order] = torch.arange(part.numel(), device=DEV) - start[part[order]]
    return rank


class _Mas:
    """The multilevel additive Schwarz preconditioner of an _Matrix in 64 bits."""

    def __init__(self, A, slot, n_slots, pairs, N, L, prec):
        self.N, self.items, self.inv = N, [slot], []
        count, real = n_slots, A.n
        while len(self.items) < L and count > N:
            it = self.items[-1]
            e = it[pairs]
            e = e[(e[:, 0] != e[:, 1]) & (e[:, 0] // N == e[:, 1] // N)]
            label = torch.arange(count, device=DEV)
            while True:
                new = label.scatter_reduce(0, e[:, 0], label[e[:, 1]], "amin").scatter_reduce(
                    0, e[:, 1], label[e[:, 0]], "amin")
                if torch.equal(new, label):
                    break
                label = new
            ids, nxt = torch.unique(label[it], return_inverse=True)
            if ids.numel() >= real:
                break
            self.items.append(nxt)
            count = real = ids.numel()
        ld = 3 * N
        k = torch.arange(3, device=DEV)
        for l, it in enumerate(self.items):
            D = -(-(n_slots if l == 0 else int(it.max()) + 1) // N)
            M = torch.zeros(D * ld * ld, dtype=F64, device=DEV)
            for r, c, b in ((A.rid, A.cid, A.au), (A.cid[A.off], A.rid[A.off], A.au[A.off].transpose(1, 2))):
                i, j = it[r], it[c]
                s = i // N == j // N
                i, j = i[s], j[s]
                at = ((i // N * ld + 3 * (i % N))[:, None, None] + k[:, None]) * ld + 3 * (j % N)[:, None, None] + k
                M.index_add_(0, at.reshape(-1), b[s].reshape(-1))
            M = M.reshape(D, ld, ld)
            pad = torch.ones(D * N, dtype=F64, device=DEV)
            pad[it] = 0.0
            pad = pad.repeat_interleave(3).reshape(D, ld)
            M = M + torch.diag_embed(pad)
            if prec == "bf16" and l == 0:  # the factor W = L^-1 rounded, as the form defines it
                W = torch.linalg.inv(torch.linalg.cholesky(M)).float().bfloat16().double()
                I = W.transpose(1, 2) @ W
            else:
                I = torch.linalg.inv(M)
            self.inv.append(I - torch.diag_embed(pad))

    def __call__(self, r):  # (n, 3, k)
        z = torch.zeros_like(r)
        for it, I in zip(self.items, self.inv):
            v = torch.zeros((I.shape[0] * self.N, 3, r.shape[2]), dtype=F64, device=DEV).index_add_(0, it, r)
            v = I @ v.reshape(I.shape[0], 3 * self.N, -1)
            z += v.reshape(-1, 3, r.shape[2])[it]
        return z


def _cg(A, M, b, iters, tol=0.0, seg=None):
    """iters steps (fewer where every column has reached tol) of PCG; seg: system of every node (one recurrence each)."""
    if seg is None:
        dot = lambda u, v: (u * v).sum((0, 1))
    else:
        S = int(seg.max()) + 1
        dot = lambda u, v: torch.zeros(S, dtype=F64, device=DEV).index_add_(0, seg, (u * v).sum((1, 2)))[seg][:, None, None]
    x, r = torch.zeros_like(b), b.clone()
    z = M(r)
    p, rz, bb = z.clone(), dot(r, z), dot(b, b)
    for _ in range(iters):
        Ap = A(p)
        al = rz / dot(p, Ap)
        x, r = x + al * p, r - al * Ap
        if bool((dot(r, r) <= tol * tol * bb).all()):
            break
        z = M(r)
        new = dot(r, z)
        p, rz = z + new / rz * p, new
    return x, torch.sqrt(dot(r, r) / bb)


def _nodes(v):
    """(k, 3n) -> (n, 3, k), and back."""
    return v.reshape(v.shape[0], -1, 3).permute(1, 2, 0).contiguous()


def _vec(x):
    return x.permute(2, 0, 1).reshape(x.shape[2], -1).contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("assemble", "abd"):
        if kind == "assemble":
            sc = _tet_scene(case, seed)[0]
            return _sum_blocks(sc.V, sc.rows, sc.cols, sc.blocks)
        return _exact_abd(_abd_scene(case, seed), case["bodies"])
    if kind == "cloth":
        X, x, tris, hinges = _sheet(case["n"], _gen(seed))
        r, c, b = _cloth_blocks(X, x, tris, hinges)
        return _i32(r), _i32(c), b
    if kind == "newton":
        return _exact_newton(case, seed)
    if kind == "batch":
        sc, off, g = _batch_scene(case, seed)
        b = _nodes(_randn((3 * sc.V,), g)[None])
        sizes = np.diff(off)
        dom = -(-sizes // case["N"])
        slot = torch.cat([_bisection(sc.X[o:o + s], case["N"]) + case["N"] * int(d)
                          for o, s, d in zip(off, sizes, np.cumsum(dom) - dom)])
        n_slots = int(dom.sum()) * case["N"]
        seg = torch.repeat_interleave(torch.arange(len(sizes), device=DEV), torch.as_tensor(sizes, device=DEV))
    else:
        sc, g = (_cloth_scene if case.get("scene") == "cloth" else _tet_scene)(case, seed)
        b = _nodes(_randn((case["nrhs"], 3 * sc.V), g))
        slot, seg = _bisection(sc.X, case["N"]), None
        n_slots = -(-sc.V // case["N"]) * case["N"]
    A = _Matrix(sc.V, sc.rows, sc.cols, sc.blocks)
    M = _Mas(A, slot, n_slots, torch.cat([sc.edges, sc.contacts]), case["N"], case["L"], case["prec"])
    if kind == "build":
        return _vec(M(b))
    if kind == "pcg":
        x, rel = _cg(A, M, b, case["iters"])
        return _vec(x), rel
    if kind == "batch":
        x, rel = _cg(A, M, b, case["iters"], seg=seg)
        return _vec(x)[0], rel.reshape(-1)[torch.as_tensor(off[:-1].astype(np.int64), device=DEV)]
    x, _ = _cg(A, M, b, 3000, 1e-13)
    if kind == "solve":
        return _vec(x)
    lam, _ = _cg(A, M, _nodes(_randn((case["nrhs"], 3 * sc.V), g)), 3000, 1e-13)
    r, c = sc.rows.long(), sc.cols.long()
    outer = lambda u, v: torch.einsum("nak,nbk->nab", u, v)
    dH = -outer(lam[r], x[c]) - torch.where((r != c)[:, None, None], outer(x[r], lam[c]), 0.0)
    return _vec(x), _vec(lam), dH


def _exact_abd(sc, bodies):
    """Every triplet mapped through J = [I, xbar_1 I, xbar_2 I, xbar_3 I], then summed per key."""
    V, nn = sc.V, sc.n_nodes
    rows, cols, blocks = sc.rows.long(), sc.cols.long(), sc.blocks
    body = torch.cat([sc.body.long(), torch.arange(4 * bodies, device=DEV) // 4])
    node = torch.arange(nn + 4 * bodies, device=DEV)
    single = (node < V) | (node >= nn)
    base = torch.where(node < V, node, torch.where(node >= nn, V + node - nn, V + 4 * body))
    w = torch.ones((node.numel(), 4), dtype=F64, device=DEV)
    w[:nn, 1:] = sc.xbar
    out = []
    for flip in (False, True):
        keep = rows != cols if flip else torch.ones_like(rows, dtype=torch.bool)
        r, c, b = (cols[keep], rows[keep], blocks[keep].transpose(1, 2)) if flip else (rows, cols, blocks)
        for a in range(4):
            ra = (a == 0) | ~single[r]
            for q in range(4):
                s = ra & ((q == 0) | ~single[c]) & (base[r] + a <= base[c] + q)
                out.append((base[r[s]] + a, base[c[s]] + q, (w[r[s], a] * w[c[s], q])[:, None, None] * b[s]))
    return _sum_blocks(V + 4 * bodies, *(torch.cat(p) for p in zip(*out)))


def _cloth_blocks(X, x, tris, hinges):
    """Stretching, strain limit, shearing, hinge bending and mass blocks, element by element."""
    E, lam, t = SHEET["E"], SHEET["lam"], SHEET["thickness"]
    d = (X[tris[:, 1:]] - X[tris[:, :1]])[:, :, :2].transpose(1, 2)  # edges as columns
    det = d[:, 0, 0] * d[:, 1, 1] - d[:, 0, 1] * d[:, 1, 0]
    inv = torch.stack([torch.stack([d[:, 1, 1], -d[:, 0, 1]], 1), torch.stack([-d[:, 1, 0], d[:, 0, 0]], 1)], 1)
    inv = inv / det[:, None, None]
    area = det.abs() / 2
    w = torch.cat([-inv.sum(1, keepdim=True), inv], 1)  # (T, 3, 2)
    F = torch.einsum("tax,tai->txi", x[tris], w)
    eye = torch.eye(3, dtype=F64, device=DEV)
    H = torch.zeros((tris.shape[0], 2, 3, 2, 3), dtype=F64, device=DEV)
    for i in range(2):
        f = F[:, :, i]
        s = f.norm(dim=1)
        ff = f[:, :, None] * f[:, None, :] / (s * s)[:, None, None]
        H[:, i, :, i, :] += 2 * lam * (ff + (1 - 1 / s).clamp_min(0)[:, None, None] * (eye - ff))
        H[:, i, :, i, :] += torch.where((s > 1)[:, None, None], 3 * E * (((1 - 1 / s) * (s - 1))[:, None, None] * eye
                                        + ((s * s - 1) / s)[:, None, None] * ff), 0.0)
    g = torch.stack([F[:, :, 1], F[:, :, 0]], 1)
    H += 0.6 * lam * g[:, :, :, None, None] * g[:, None, None, :, :]
    H *= (area * t)[:, None, None, None, None]
    out = []

    def emit(elements, blocks):  # (E, pairs, 3, 3) in the pair order a <= b
        k = elements.shape[1]
        a, b = torch.tensor([(p, q) for p in range(k) for q in range(p, k)], device=DEV).T
        r, c = elements[:, a], elements[:, b]
        blocks = torch.where((r > c)[..., None, None], blocks.transpose(-1, -2), blocks)
        out.append((torch.minimum(r, c).reshape(-1), torch.maximum(r, c).reshape(-1), blocks.reshape(-1, 3, 3)))

    emit(tris, torch.stack([torch.einsum("ti,tj,tixjy->txy", w[:, a], w[:, b], H) for a in range(3) for b in range(a, 3)], 1))
    with torch.enable_grad():  # gradient of the dihedral angle
        P = x[hinges].clone().requires_grad_(True)
        e = P[:, 1] - P[:, 0]
        n1 = torch.linalg.cross(e, P[:, 2] - P[:, 0], dim=1)
        n2 = torch.linalg.cross(P[:, 3] - P[:, 0], e, dim=1)
        theta = torch.atan2((torch.linalg.cross(n1, n2, dim=1) * e).sum(1) / e.norm(dim=1), (n1 * n2).sum(1))
        gr, = torch.autograd.grad(theta.sum(), P)
    e = X[hinges[:, 1]] - X[hinges[:, 0]]
    A12 = sum(torch.linalg.cross(e, X[hinges[:, q]] - X[hinges[:, 0]], dim=1).norm(dim=1) / 2 for q in (2, 3))
    kb = E * t ** 3 / 12 * (e * e).sum(1) / A12
    emit(hinges, torch.stack([2 * kb[:, None, None] * gr[:, a, :, None] * gr[:, b, None, :]
                              for a in range(4) for b in range(a, 4)], 1))
    m = torch.zeros(X.shape[0], dtype=F64, device=DEV)
    m.index_put_((tris.reshape(-1),), (SHEET["rho"] * t * area / 3).repeat_interleave(3), accumulate=True)
    v = torch.arange(X.shape[0], device=DEV)
    out.append((v, v, (m / DT ** 2)[:, None, None] * eye))
    return tuple(torch.cat(p) for p in zip(*out))


def _exact_newton(case, seed):
    """Newton's method on the step's potential with eigenvalue-clamped element Hessians and exact directions."""
    X, x, xt, tets, pairs, K = _elastic_scene(case, seed)
    V, E = X.shape[0], case["E"]
    vol, w = _weights(X, tets)
    mu_l, lam_l = E / (2 * (1 + NU)), E * NU / ((1 + NU) * (1 - 2 * NU))
    mu, lam = 4 / 3 * mu_l, lam_l + 5 / 6 * mu_l
    alpha = 1 + mu / lam
    mr, _, mb = (t[-V:] for t in _tet_triplets(X, tets, E))
    m = mb[:, 0, 0]  # m / dt^2
    rest = X[pairs[:, 0]] - X[pairs[:, 1]]
    eps = torch.zeros((3, 3, 3), dtype=F64, device=DEV)
    eps[[0, 1, 2], [1, 2, 0], [2, 0, 1]], eps[[0, 1, 2], [2, 0, 1], [1, 2, 0]] = 1.0, -1.0
    pa, pb = (torch.tensor(p, device=DEV) for p in zip(*_PAIRS4))
    r, c = tets[:, pa], tets[:, pb]
    slot, n_slots = _bisection(X, case["N"]), -(-V // case["N"]) * case["N"]
    edges = torch.cat([_edges(tets), pairs])

    def energy(y):
        F = torch.einsum("tax,taj->txj", y[tets], w)
        J = torch.linalg.det(F)
        d = y[pairs[:, 0]] - y[pairs[:, 1]] - rest
        return ((vol * (mu / 2 * ((F * F).sum((1, 2)) - 3) + lam / 2 * (J - alpha) ** 2)).sum()
                + (m[:, None] * (y - xt) ** 2).sum() / 2 + 0.5 * torch.einsum("px,pxy,py->", d, K, d))

    for _ in range(case["steps"]):
        with torch.enable_grad():
            y = x.clone().requires_grad_(True)
            g, = torch.autograd.grad(energy(y), y)
        F = torch.einsum("tax,taj->txj", x[tets], w)
        J = torch.linalg.det(F)
        co = 0.5 * torch.einsum("xyz,ijk,tyj,tzk->txi", eps, eps, F, F)  # dJ / dF
        H = lam * co[:, :, :, None, None] * co[:, None, None]
        H += (lam * (J - alpha))[:, None, None, None, None] * torch.einsum("xyz,ijk,tzk->txiyj", eps, eps, F)
        H = H.reshape(-1, 9, 9) + mu * torch.eye(9, dtype=F64, device=DEV)
        for i in range(0, H.shape[0], 16384):
            ev, Q = torch.linalg.eigh(H[i:i + 16384])
            H[i:i + 16384] = (Q * ev.clamp_min(0)[:, None, :]) @ Q.transpose(1, 2)
        Hw = torch.einsum("txiyj,taj->taxiy", H.reshape(-1, 3, 3, 3, 3), w)  # [t, b, x, i, y]
        blk = torch.stack([torch.einsum("ti,txiy->txy", w[:, a], Hw[:, b]) for a, b in _PAIRS4], 1)
        blk *= vol[:, None, None, None]
        blk = torch.where((r > c)[..., None, None], blk.transpose(-1, -2), blk)
        trip = [(torch.minimum(r, c).reshape(-1), torch.maximum(r, c).reshape(-1), blk.reshape(-1, 3, 3)), (mr, mr, mb),
                _contact_triplets(pairs, K)]
        A = _Matrix(V, *(torch.cat(p) for p in zip(*trip)))
        M = _Mas(A, slot, n_slots, edges, case["N"], case["L"], "fp64")
        x = x - _cg(A, M, g[:, :, None], 1000, 1e-12)[0][:, :, 0]
    return x, np.float64(energy(x).item())
