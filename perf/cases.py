"""Timed cases of the framework: what its users have it do, through the public calls.

A case is a dict of plain values; ``kind`` says which call it times:

* ``solve``   -- a whole molecule: pb_mesh_upload, pb_build_tree, pb_gmres_solve and the energy,
* ``product`` -- pb_matvec, the operator every solver iteration applies (constant or linear basis),
* ``multi``   -- pb_matvec_multi, the same operator on the charge states of a titration at once,
* ``precond`` -- pb_precond_apply,
* ``source``  -- pb_rhs and the treecode energy: the two passes over charges x elements,
* ``train``   -- pb_mlp_gradient, one mini-batch of the learned start's training.

Surfaces are seeded: a geodesic sphere of 20 n^2 triangles with jittered vertices and random bumps
at the benchmark's element size (about 0.35 A^2, so 1.8 M triangles would be its 20,000-atom
molecule), the plain sphere of the Kirkwood benchmark (radius 20 A), or a protein-like molecule of
``molecules.molecule`` (marching tetrahedra, short edges collapsed: ragged triangles and odd counts).
Parameters are the benchmark's (eps 1 / 80, kappa 0.1257, eta0 0.8, leaf 64, order 8) unless a
case says otherwise.
"""
import functools
import math

import numpy as np
import torch

from paper_2110_13778_gb300 import inputs, molecules, pb

AREA = 0.35  # A^2 per triangle of the bumpy surfaces
TOL = 1e-6
DENSE_PAIRS = 7e9  # point pairs that exact() sums in a few seconds
DENSE_SOLVE = 6000  # elements of the largest system that exact() factors


def listed():
    return [
        # the smallest molecule a user solves (the Kirkwood check): launches and latency
        {"name": "solve_1280", "kind": "solve", "shape": "sphere", "n": 8, "charges": 5, "restart": 50,
         "energy": "direct"},
        # a large protein start to finish, the benchmark's step: upload, build, solve, treecode energy
        {"name": "solve_1310720", "kind": "solve", "shape": "bumpy", "n": 256, "charges": 14000, "restart": 200,
         "energy": "tree"},
        # one product on the smallest mesh: latency
        {"name": "product_1280", "kind": "product", "shape": "sphere", "n": 8},
        # one product on a small protein: marching-tetrahedra triangles, an odd count
        {"name": "product_molecule200", "kind": "product", "shape": "molecule", "n": 200},
        # the Kirkwood benchmark's sphere at its finest mesh
        {"name": "product_81920", "kind": "product", "shape": "sphere", "n": 64},
        # one product on a large protein: throughput
        {"name": "product_737280", "kind": "product", "shape": "bumpy", "n": 192},
        # the default precision of the parameters: the reference product users check against
        {"name": "product_fp64_20480", "kind": "product", "shape": "bumpy", "n": 32, "precision": "fp64"},
        # the hat-function basis with the order-2 rule
        {"name": "product_linear_20480", "kind": "product", "shape": "bumpy", "n": 32, "basis": "linear", "qr": 2},
        # 16 charge states of one protein in lockstep, as the batched solve applies them
        {"name": "multi16_81920", "kind": "multi", "shape": "bumpy", "n": 64, "nr": 16},
        # the block-diagonal preconditioner of every iteration
        {"name": "precond_327680", "kind": "precond", "shape": "bumpy", "n": 128},
        # right-hand side and energy of a mid-size protein (charges x elements)
        {"name": "source_81920", "kind": "source", "shape": "bumpy", "n": 64, "charges": 900},
        # a mini-batch of the learned start's training at its default size
        {"name": "train_4096", "kind": "train", "rows": 4096},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "product", "product", "product", "multi", "precond", "source", "train"])
    if kind == "train":
        return {"kind": kind, "rows": _log(rng, 500, 16384)}
    c = {"kind": kind, "shape": rng.choice(["sphere", "bumpy", "bumpy", "molecule"]), "n": _log(rng, 8, 190),
         "leaf": rng.choice([48, 64, 64, 80]), "p": rng.choice([4, 6, 8, 8]),
         "kappa": round(rng.uniform(0.03, 0.3), 4), "eta0": rng.choice([0.7, 0.8])}
    if c["shape"] == "molecule":
        c["n"] = _log(rng, 20, 400)  # atoms; about 100 triangles each
    elif c["shape"] == "sphere":
        c["n"] = min(c["n"], 100)
    if kind in ("solve", "source") and c["shape"] != "molecule":  # a molecule's charges are its atoms
        c["charges"] = _log(rng, 5, 2500)
    if kind == "solve":
        c["restart"] = rng.choice([30, 50, 200])
        c["energy"] = rng.choice(["direct", "tree"])
    elif kind == "multi":
        c["n"] = min(c["n"], 90) if c["shape"] != "molecule" else c["n"]
        c["nr"] = rng.randint(2, 20)
    elif kind == "product":
        form = rng.choice(["mixed", "mixed", "fp64", "linear", "order2"])
        if form != "mixed" and c["shape"] != "molecule":
            c["n"] = min(c["n"], 40)
        if form == "fp64":
            c["precision"] = "fp64"
        elif form == "linear":
            c["basis"], c["qr"] = "linear", 2
        elif form == "order2":
            c["qr"] = 2
    return c


# ---------------- inputs ----------------
@functools.lru_cache(maxsize=2)
def _geodesic(n):
    """Unit geodesic sphere: every icosahedron face cut into n^2 triangles (the topology only depends on n)."""
    V, F = inputs.icosphere(0)
    i, j = np.meshgrid(np.arange(n + 1), np.arange(n + 1), indexing="ij")
    keep = i + j <= n
    i, j = i[keep], j[keep]  # barycentric grid points of one face
    at = np.full((n + 1, n + 1), -1)
    at[i, j] = np.arange(i.size)
    up = np.argwhere(np.add.outer(np.arange(n), np.arange(n)) < n)
    dn = up[up.sum(1) < n - 1]
    T = np.concatenate([
        np.stack([at[up[:, 0], up[:, 1]], at[up[:, 0] + 1, up[:, 1]], at[up[:, 0], up[:, 1] + 1]], 1),
        np.stack([at[dn[:, 0] + 1, dn[:, 1]], at[dn[:, 0] + 1, dn[:, 1] + 1], at[dn[:, 0], dn[:, 1] + 1]], 1)])
    w = np.stack([n - i - j, i, j], 1)  # integer barycentric weights
    P, K = [], []
    for f in F:
        P.append(w @ V[f] / n)
        # a point is known by its weights on the icosahedron's vertices, sorted by vertex
        o = np.argsort(f)
        fs, ws = f[o].astype(np.int64), w[:, o].astype(np.int64)
        k = np.zeros((w.shape[0], 3), np.int64)
        for a in range(3):
            k[:, a] = np.where(ws[:, a] > 0, fs[a] * (n + 1) + ws[:, a], -1)
        k = np.sort(k, 1) + 1
        b = 12 * (n + 1) + 1
        K.append((k[:, 2] * b + k[:, 1]) * b + k[:, 0])
    K = np.concatenate(K)
    _, first, inv = np.unique(K, return_index=True, return_inverse=True)
    U = np.concatenate(P)[first]
    U /= np.linalg.norm(U, axis=1, keepdims=True)
    tris = inv[np.concatenate([T + s * i.size for s in range(len(F))])]
    A = U[tris]
    out = np.einsum("ij,ij->i", np.cross(A[:, 1] - A[:, 0], A[:, 2] - A[:, 0]), A[:, 0]) > 0
    tris = np.where(out[:, None], tris, tris[:, [0, 2, 1]])
    return U, tris.astype(np.int32)


@functools.lru_cache(maxsize=2)
def _molecule(n):
    return molecules.molecule(n, 5000 + n, 0.9, clean=True)[0]


def _mesh(case, seed):
    """(verts, tris, charge positions, charges) of the case, from the seed alone."""
    rng = np.random.default_rng([seed, 211])
    n, nc = case["n"], case.get("charges", 1)
    if case["shape"] == "molecule":
        # one molecule per size (so that its counts stay), turned, moved and scaled by up to 2 %
        m = _molecule(n)
        Q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        Q = Q * np.sign(np.linalg.det(Q)) * rng.uniform(0.98, 1.02)
        b = rng.uniform(-5.0, 5.0, size=3)
        return m.verts @ Q + b, m.tris, m.qpos @ Q + b, rng.permutation(m.q)
    U, T = _geodesic(n)
    d = rng.normal(size=(nc, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    if case["shape"] == "sphere":
        V, r = 20.0 * U if n > 16 else 2.0 * U, (16.0 if n > 16 else 1.5)
    else:
        # jittered directions, then radial bumps of 0.2 to 0.7 rad
        e = math.sqrt(4 * math.pi / T.shape[0] * 2.3)
        W = U + rng.uniform(-0.12, 0.12, size=U.shape) * e
        W /= np.linalg.norm(W, axis=1, keepdims=True)
        R = math.sqrt(T.shape[0] * AREA / (4 * math.pi))
        c = rng.normal(size=(24, 3))
        c /= np.linalg.norm(c, axis=1, keepdims=True)
        h, s = rng.uniform(-0.06, 0.12, size=24), rng.uniform(4.0, 30.0, size=24)
        rad = 1.0 + (h * np.exp(s * (W @ c.T - 1.0))).sum(1)
        V, r = W * (R * rad)[:, None], 0.8 * R * float(rad.min())
        V = V + rng.uniform(-5.0, 5.0, size=3)
    pos = d * (r * rng.uniform(0.0, 1.0, size=nc) ** (1.0 / 3.0))[:, None]
    if case["shape"] == "bumpy":
        pos = pos + V.mean(0)
    return V, T, pos, rng.uniform(-0.8, 0.8, size=nc)


def _vector(case, n, seed, nr=None):
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed % 100000) + 17)
    return torch.rand((n,) if nr is None else (nr, n), generator=g, device="cuda", dtype=torch.float64) * 2 - 1


def _params(case):
    return pb.params(eta0=case.get("eta0", 0.8), leaf_size=case.get("leaf", 64), p=case.get("p", 8),
                     kappa=case.get("kappa", 0.1257), qr=case.get("qr", 0),
                     precision=pb.PB_FP64 if case.get("precision") == "fp64" else pb.PB_MIXED,
                     basis=pb.PB_BASIS_LINEAR if case.get("basis") == "linear" else pb.PB_BASIS_CONSTANT)


class _State:
    """What a program holds: the context (destroyed with it), its mesh and its vectors."""

    def __init__(self, case):
        self.case, self.ctx, self.net = case, None, None

    def __del__(self):
        if self.ctx is not None:
            pb.pb_destroy(self.ctx)
        if self.net is not None:
            pb.pb_mlp_destroy(self.net)


def _weights(seed):
    """Network parameters in the library's padded layout (18 -> 128 x 3 -> 2, padded to 32 and 16)."""
    rng = np.random.default_rng([seed, 7])
    W, B = [], []
    for fin, fout, pin, pout in ((18, 128, 32, 128), (128, 128, 128, 128), (128, 128, 128, 128), (128, 2, 128, 16)):
        w = np.zeros((pout, pin), np.float32)
        w[:fout, :fin] = rng.uniform(-1, 1, size=(fout, fin)) * math.sqrt(6.0 / (fin + fout))
        b = np.zeros(pout, np.float32)
        b[:fout] = rng.uniform(-0.05, 0.05, size=fout)
        W.append(w)
        B.append(b)
    return W, B


def _rows(case, seed):
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed % 100000) + 29)
    X = torch.randn((case["rows"], pb.NFEAT), generator=g, device="cuda")
    T = torch.randn((case["rows"], 2), generator=g, device="cuda")
    return X, T


def prepare(case, seed):
    s = _State(case)
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "train":
        s.X, s.T = _rows(case, seed)
        s.net = pb.pb_mlp_create(pb.NFEAT, 128, 3, 2, seed=17, stream=stream)
        W, B = _weights(seed)
        pb.pb_mlp_set_params(s.net, np.concatenate([a.ravel() for a in W + B]))
        return s
    s.mesh = _mesh(case, seed)
    s.ctx = pb.pb_create(_params(case), stream)
    nu = s.mesh[0].shape[0] if case.get("basis") == "linear" else s.mesh[1].shape[0]
    if case["kind"] == "solve":
        s.y = torch.zeros(2 * nu, device="cuda", dtype=torch.float64)
        return s  # the mesh is uploaded and built by the timed call
    pb.pb_mesh_upload(s.ctx, *s.mesh)
    pb.pb_build_tree(s.ctx)
    s.x = _vector(case, 2 * nu, seed, case.get("nr"))
    s.y = torch.empty_like(s.x)
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "product":
        pb.pb_matvec(s.ctx, s.x, s.y)
        return s.y
    if kind == "multi":
        pb.pb_matvec_multi(s.ctx, s.x, s.y)
        return s.y
    if kind == "precond":
        pb.pb_precond_apply(s.ctx, s.x, s.y)
        return s.y
    if kind == "source":
        pb.pb_rhs(s.ctx, s.y)
        return s.y, pb.pb_solvation_energy_treecode(s.ctx, s.x)
    if kind == "train":
        return pb.pb_mlp_gradient(s.net, s.X, s.T)
    pb.pb_mesh_upload(s.ctx, *s.mesh)
    pb.pb_build_tree(s.ctx)
    info = pb.pb_gmres_solve(s.ctx, s.y, tol=TOL, max_iter=400, restart=s.case["restart"])
    tree = s.case["energy"] == "tree"
    return s.y, info.iterations, (pb.pb_solvation_energy_treecode if tree else pb.pb_solvation_energy)(s.ctx, s.y)


def work(case):
    """Sizes from the method: about 27 neighbour leaves and 25 interactions per leaf, 75 flops per
    element pair, 2 C(p + 6, 6) per cluster pair and kernel."""
    if case["kind"] == "train":
        r = case["rows"]
        return {"bytes": 4.0 * r * 20 + 8.0 * 39000, "flops": 6.0 * r * (18 * 128 + 2 * 128 * 128 + 128 * 2)}
    N = 100.0 * case["n"] if case["shape"] == "molecule" else 20.0 * case["n"] ** 2
    leaf, p, q2 = case.get("leaf", 64), case.get("p", 8), max(1, case.get("qr", 1)) ** 2
    near = N * min(N, 27.0 * leaf)
    far = 4.0 * math.comb(p + 6, 6) * 25 * 1.33 * N / leaf if N > 27 * leaf else 0.0
    nr = case.get("nr", 1)
    flops = 75.0 * near * q2 * q2 + far + 8.0 * near * (nr - 1) + far * (nr - 1)
    geometry, vectors = 96.0 * N, 32.0 * N * nr
    blocks = 4.0 * 4 * 70 * N  # the inverse blocks of leaves of about 70 elements, FP32
    corr = 36.0 * 13.3 * N
    if case["kind"] == "precond":
        return {"bytes": blocks + vectors, "flops": blocks / 2}
    nc = case["n"] if case["shape"] == "molecule" else case.get("charges", 1)
    source = 20.0 * N * nc
    if case["kind"] == "source":
        return {"bytes": geometry + vectors, "flops": source}
    if case["kind"] == "solve":  # about ten iterations, and the touching pairs' integrals once
        return {"bytes": 10 * (geometry + corr + blocks) + 10 * 55 * 16.0 * N,
                "flops": 10 * flops + source + 6.6 * N * 400 * 100.0}
    return {"bytes": geometry + corr + vectors, "flops": flops}


# ---------------- the same in 64 bits ----------------
I4PI = 1.0 / (4.0 * math.pi)


def _kernels(d, nx, ny, eps, kappa):
    """K1..K4 of the derivative boundary integral equations; d = x - y, nx, ny broadcast against it."""
    r2 = (d * d).sum(-1)
    ri = torch.where(r2 > 0, r2, torch.ones_like(r2)).rsqrt()
    t = kappa * r2 * ri
    e = torch.exp(-t)
    xd, yd = (nx * d).sum(-1), (ny * d).sum(-1)
    g3 = I4PI * ri ** 3
    k1 = -torch.expm1(-t) * ri * I4PI
    k2 = yd * g3 * (eps * e * (1 + t) - 1)
    k3 = -xd * g3 * (1 - e * (1 + t) / eps)
    k4 = g3 * ((3 - e * (3 + 3 * t + t * t)) * xd * yd * ri * ri - (1 - e * (1 + t)) * (nx * ny).sum(-1))
    return k1, k2, k3, k4


def _dense_rows(P, Nn, W, f, eps, kappa):
    """Sums over all points y of W_y [K1 f2 + K2 f1] and W_y [K3 f2 + K4 f1] at all points x (f: (2, points, nr))."""
    M = P.shape[0]
    o1, o2 = torch.zeros_like(f[0]), torch.zeros_like(f[0])
    g1, g2 = W[:, None] * f[0], W[:, None] * f[1]
    at = torch.arange(M, device=P.device)
    step = max(1, int(6e7) // M)
    for a in range(0, M, step):
        b = min(M, a + step)
        dx, dy, dz = (P[a:b, None, k] - P[None, :, k] for k in range(3))
        r2 = dx * dx + dy * dy + dz * dz
        r2[at[a:b] - a, at[a:b]] = 1.0
        ri = r2.rsqrt()
        t = kappa * r2 * ri
        e = torch.exp(-t)
        xd = Nn[a:b, None, 0] * dx + Nn[a:b, None, 1] * dy + Nn[a:b, None, 2] * dz
        yd = Nn[None, :, 0] * dx + Nn[None, :, 1] * dy + Nn[None, :, 2] * dz
        del dx, dy, dz, r2
        g = I4PI * ri
        g[at[a:b] - a, at[a:b]] = 0.0
        e1 = e * (1 + t)
        o1[a:b] = (-torch.expm1(-t) * g) @ g2
        g = g * ri * ri
        o1[a:b] += (yd * g * (eps * e1 - 1)) @ g1
        o2[a:b] = (-xd * g * (1 - e1 / eps)) @ g2
        c3 = 3 - e * (3 + 3 * t + t * t)
        o2[a:b] += (g * (c3 * xd * yd * ri * ri - (1 - e1) * (Nn[a:b] @ Nn.T))) @ g1
    return o1, o2


def _touching(T, nv):
    """Ordered pairs of elements i <= j that share 1, 2 or 3 vertices, by that number, each with its corners
    turned so that the shared ones come first, in i's order."""
    nt = T.shape[0]
    flat = T.reshape(-1)
    o = np.argsort(flat, kind="stable")
    start = np.searchsorted(flat[o], np.arange(nv + 1))
    deg = np.diff(start)
    a, b = [], []
    for k in range(int(deg.max())):
        for m in range(int(deg.max())):
            v = np.flatnonzero((deg > k) & (deg > m))
            a.append(o[start[v] + k] // 3)
            b.append(o[start[v] + m] // 3)
    a, b = np.concatenate(a).astype(np.int64), np.concatenate(b).astype(np.int64)
    key = np.unique((a * nt + b)[a < b])
    i, j = key // nt, key % nt
    eq = T[i][:, :, None] == T[j][:, None, :]
    shared = eq.any(2).sum(1)
    out = {3: (np.arange(nt), np.arange(nt), np.tile([0, 1, 2], (nt, 1)), np.tile([0, 1, 2], (nt, 1)))}
    for c in (1, 2):
        s = np.flatnonzero(shared == c)
        e = eq[s]
        ci = np.argsort(~e.any(2), axis=1, kind="stable")  # shared corners of i first, then the others in order
        mate = np.take_along_axis(np.argmax(e, axis=2), ci, 1)
        cj = np.zeros_like(ci)
        cj[:, :c] = mate[:, :c]
        rest = np.ones((s.size, 3), bool)
        np.put_along_axis(rest, cj[:, :c], False, 1)
        cj[:, c:] = np.argsort(~rest, axis=1, kind="stable")[:, :3 - c]
        out[c] = (i[s], j[s], ci, cj)
    return out


def _cube(shared, qs):
    """Sauter-Schwab points (x1, x2, y1, y2, weight) of two triangles sharing that many vertices (Section 3 of
    the method; reference triangle 0 <= e2 <= e1 <= 1)."""
    g, w = np.polynomial.legendre.leggauss(qs)
    g, w = (g + 1) / 2, w / 2
    z, a, b, c = (x.ravel() for x in np.meshgrid(g, g, g, g, indexing="ij"))
    wt = np.prod(np.meshgrid(w, w, w, w, indexing="ij"), axis=0).ravel()
    one = np.ones_like(z)
    if shared == 1:
        jac = [z ** 3 * b] * 2
        pts = [(one, a, b, b * c), (b, b * a, one, c)]
    elif shared == 2:
        jac = [z ** 3 * a ** 2] + [z ** 3 * a ** 2 * b] * 4
        pts = [(one, a * c, 1 - a * b, a * (1 - b)), (one, a, 1 - a * b * c, a * b * (1 - c)),
               (1 - a * b, a * (1 - b), one, a * b * c), (1 - a * b * c, a * b * (1 - c), one, a),
               (1 - a * b * c, a * (1 - b * c), one, a * b)]
    else:
        jac = [z ** 3 * a ** 2 * b] * 6
        pts = [(one, 1 - a + a * b, 1 - a * b * c, 1 - a), (1 - a * b * c, 1 - a, one, 1 - a + a * b),
               (one, a * (1 - b + b * c), 1 - a * b, a * (1 - b)), (1 - a * b, a * (1 - b), one, a * (1 - b + b * c)),
               (1 - a * b * c, a * (1 - b * c), one, a * (1 - b)), (one, a * (1 - b), 1 - a * b * c, a * (1 - b * c))]
    rows = [np.stack([z * x for x in p] + [wt * j], 1) for p, j in zip(pts, jac)]
    return np.concatenate(rows)


def _hat(e1, e2):
    return torch.stack([1 - e1, e1 - e2, e2], -1)


def _rule(q):
    """Points of the order-q rule on the reference triangle and their weights (sum 1/2)."""
    if q == 1:
        return np.array([2 / 3]), np.array([1 / 3]), np.array([0.5])
    k, m = np.arange(q), np.arange(1, q)
    J = np.diag((1.0 / ((2 * k + 1) * (2 * k + 3)) + 1) / 2)
    off = np.sqrt(m * (m + 1) / (2.0 * m + 1) ** 2 / 4)
    t, U = np.linalg.eigh(J + np.diag(off, 1) + np.diag(off, -1))
    g, w = np.polynomial.legendre.leggauss(q)
    return (np.repeat(t, q), np.repeat(t, q) * np.tile((g + 1) / 2, q), np.outer(0.5 * U[0] ** 2, w / 2).ravel())


class _Exact:
    """The discretised operator in plain torch FP64: regular rule, Sauter-Schwab for touching pairs, mass terms."""

    def __init__(self, case, mesh):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        V, T = mesh[0], mesh[1].astype(np.int64)
        self.linear, self.kappa, self.eps = case.get("basis") == "linear", case.get("kappa", 0.1257), 80.0
        self.T = torch.as_tensor(T, device=dev)
        self.nv, self.nt = V.shape[0], T.shape[0]
        self.C = torch.as_tensor(V, device=dev, dtype=torch.float64)[self.T]  # corners (nt, 3, 3)
        c = torch.linalg.cross(self.C[:, 1] - self.C[:, 0], self.C[:, 2] - self.C[:, 0])
        self.A = c.norm(dim=1) / 2
        self.nrm = c / (2 * self.A[:, None])
        e1, e2, w = (torch.as_tensor(a, device=dev) for a in _rule(max(1, case.get("qr", 1))))
        self.q2, self.lam = w.numel(), _hat(e1, e2)
        self.P = torch.einsum("ai,tik->tak", self.lam, self.C).reshape(-1, 3)
        self.Pn = self.nrm.repeat_interleave(self.q2, 0)
        self.W = (2 * self.A[:, None] * w[None, :]).reshape(-1)
        self.pairs = {k: [torch.as_tensor(a, device=dev) for a in v] for k, v in _touching(T, self.nv).items()}
        self.cube = {k: torch.as_tensor(_cube(k, 3), device=dev) for k in (1, 2, 3)}

    def corners(self, x):
        """(nt, 3, nr) corner values of each element."""
        return x[self.T] if self.linear else x[:, None, :].expand(-1, 3, -1)

    def product(self, x):
        """A x for x (2, unknowns, nr): rows of the two equations, the same shape."""
        f = [self.corners(x[0]), self.corners(x[1])]
        fq = torch.stack([torch.einsum("ai,tir->tar", self.lam, g).reshape(-1, g.shape[2]) for g in f])
        s1, s2 = _dense_rows(self.P, self.Pn, self.W, fq, self.eps, self.kappa)
        out = [self.test((self.W[:, None] * s).reshape(self.nt, self.q2, -1)) for s in (s1, s2)]
        self.touching(f, fq, out)
        if self.linear:
            mass = [(self.A[:, None, None] / 12) * (g + g.sum(1, keepdim=True)) for g in f]
        else:
            mass = [self.A[:, None, None] * g[:, :1] for g in f]
        m1, m2 = self.gather(mass[0]), self.gather(mass[1])
        return torch.stack([0.5 * (1 + self.eps) * m1 - self.gather(out[0]),
                            0.5 * (1 + 1 / self.eps) * m2 - self.gather(out[1])])

    def test(self, s):
        return torch.einsum("ai,tar->tir", self.lam, s) if self.linear else s.sum(1, keepdim=True)

    def gather(self, c):
        if not self.linear:
            return c[:, 0]
        out = torch.zeros((self.nv, c.shape[2]), device=c.device, dtype=c.dtype)
        return out.index_add_(0, self.T.reshape(-1), c.reshape(-1, c.shape[2]))

    def touching(self, f, fq, out):
        """Adds, for every touching pair, the Sauter-Schwab integrals minus the regular rule's."""
        nr = fq.shape[2]
        for c, (I, J, ci, cj) in self.pairs.items():
            cube = self.cube[c]
            lx, ly = _hat(cube[:, 0], cube[:, 1]), _hat(cube[:, 2], cube[:, 3])
            step = max(1, int(3e6) // (cube.shape[0] * max(1, nr // 4)))
            for a in range(0, I.numel(), step):
                i, j, pi, pj = (v[a:a + step] for v in (I, J, ci, cj))
                Ci = torch.gather(self.C[i], 1, pi[:, :, None].expand(-1, -1, 3))
                Cj = torch.gather(self.C[j], 1, pj[:, :, None].expand(-1, -1, 3))
                X, Y = torch.einsum("sq,tqk->tsk", lx, Ci), torch.einsum("sq,tqk->tsk", ly, Cj)
                w = cube[None, :, 4] * (4 * self.A[i] * self.A[j])[:, None]
                sides = [(i, j, pi, pj, X, Y, lx, ly)] + ([(j, i, pj, pi, Y, X, ly, lx)] if c < 3 else [])
                for t, s, pt, ps, x, y, hx, hy in sides:
                    nx, ny = self.nrm[t][:, None], self.nrm[s][:, None]
                    k = _kernels(x - y, nx, ny, self.eps, self.kappa)
                    g = [torch.einsum("sq,tqr->tsr", hy, torch.gather(v[s], 1, ps[:, :, None].expand(-1, -1, nr)))
                         for v in f]
                    for m in (0, 1):
                        v = (w * k[2 * m])[:, :, None] * g[1] + (w * k[2 * m + 1])[:, :, None] * g[0]
                        if self.linear:
                            v = torch.einsum("sq,tsr->tqr", hx, v)
                            v = torch.zeros_like(v).scatter_(1, pt[:, :, None].expand(-1, -1, nr), v)
                        else:
                            v = v.sum(1, keepdim=True)
                        out[m].index_add_(0, t, v)
                    # take the regular rule's sum for this pair off again (the dense sum held it, but for the
                    # terms of one point with itself)
                    q2 = self.q2
                    pq = torch.arange(q2, device=i.device)
                    xt, ys = t[:, None] * q2 + pq, s[:, None] * q2 + pq
                    d = self.P[xt][:, :, None] - self.P[ys][:, None]
                    k = _kernels(d, nx[:, :, None], ny[:, :, None], self.eps, self.kappa)
                    wq = self.W[xt][:, :, None] * self.W[ys][:, None]
                    if c == 3:
                        wq = wq * (1 - torch.eye(q2, device=i.device, dtype=wq.dtype))
                    for m in (0, 1):
                        v = torch.einsum("tab,tbr->tar", wq * k[2 * m], fq[1][ys]) + \
                            torch.einsum("tab,tbr->tar", wq * k[2 * m + 1], fq[0][ys])
                        out[m].index_add_(0, t, -self.test(v))

    def source(self, pos, q):
        """Right-hand side (2, nt) of the charges."""
        d = self.P[:, None] - torch.as_tensor(pos, device=self.P.device)[None]
        ri = d.norm(dim=2).reciprocal()
        q = torch.as_tensor(q, device=self.P.device)
        b1 = (ri * q).sum(1) * I4PI * self.W
        b2 = -(ri ** 3 * q * (d * self.Pn[:, None]).sum(2)).sum(1) * I4PI * self.W
        return torch.stack([v.reshape(self.nt, self.q2).sum(1) for v in (b1, b2)])

    def energy(self, pos, q, x):
        """Solvation energy in kcal/mol of x (2, nt): the direct sum."""
        e = torch.zeros((), device=self.P.device, dtype=torch.float64)
        f = [v.repeat_interleave(self.q2) * self.W for v in x]
        for a in range(0, len(q), 64):
            p = torch.as_tensor(pos[a:a + 64], device=self.P.device)
            k1, k2, _, _ = _kernels(p[:, None] - self.P[None], self.Pn[None], self.Pn[None], self.eps, self.kappa)
            e = e + torch.as_tensor(q[a:a + 64], device=self.P.device) @ (k1 @ f[1] + k2 @ f[0])
        return float(e) * 0.5 * 4 * math.pi * 332.0716


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        W, B = ([torch.tensor(a, device="cuda", dtype=torch.float64, requires_grad=True) for a in v]
                for v in _weights(seed))
        X, T = _rows(case, seed)
        h = torch.nn.functional.pad(X.double(), (0, 14))
        for k in range(4):
            h = h @ W[k].T + B[k]
            h = h.relu() if k < 3 else h
        loss = ((h[:, :2] - T.double()) ** 2).mean()
        g = torch.autograd.grad(loss, W + B)
        return float(loss.detach()), np.concatenate([v.cpu().numpy().ravel() for v in g])
    if kind == "precond":
        return None  # its blocks are the tree's leaves: no value without the framework's own tree
    mesh = _mesh(case, seed)
    N, q2 = mesh[1].shape[0], max(1, case.get("qr", 1)) ** 2
    if kind == "source":
        op = _Exact(case, mesh)
        x = _vector(case, 2 * N, seed).reshape(2, N)
        chunks = [op.source(mesh[2][a:a + 100], mesh[3][a:a + 100]) for a in range(0, len(mesh[3]), 100)]
        return sum(chunks).reshape(-1), op.energy(mesh[2], mesh[3], x)
    if kind == "solve":
        if N > DENSE_SOLVE:
            return None
        op = _Exact(case, mesh)
        A = torch.empty((2 * N, 2 * N), device="cuda", dtype=torch.float64)
        for a in range(0, 2 * N, 512):
            x = torch.zeros((2 * N, min(512, 2 * N - a)), device="cuda", dtype=torch.float64)
            x[torch.arange(a, a + x.shape[1]), torch.arange(x.shape[1])] = 1.0
            A[:, a:a + x.shape[1]] = op.product(x.reshape(2, N, -1)).reshape(2 * N, -1)
        x = torch.linalg.solve(A, op.source(mesh[2], mesh[3]).reshape(-1))
        return x, None, op.energy(mesh[2], mesh[3], x.reshape(2, N))
    if (float(N) * q2) ** 2 > DENSE_PAIRS:
        return None
    nu = mesh[0].shape[0] if case.get("basis") == "linear" else N
    x = _vector(case, 2 * nu, seed, case.get("nr"))
    f = x.reshape(-1, 2, nu).permute(1, 2, 0)
    return _Exact(case, mesh).product(f).permute(2, 0, 1).reshape(x.shape)
