"""Products and solutions of mixed precision keep their bits.

The FP32 block preconditioner rounds its input, so one changed last bit of a product moves single
entries of a solution by a whole FP32 ulp (1e-7 of its maximum). The digests below are those of the
kernels whose row roundings (mass term, corrections) were left to the compiler, before the passes that
end a product were fused; meshes, vectors and charges are made with exactly rounded operations, so that
they are the same on every machine. A change of the compiler or of the FP32 evaluation moves them."""
import hashlib

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2110_13778_gb300 import inputs, pb  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2110_13778_gb300 import build

    build.build()
    pb.lib()


def octasphere(k, radii=(9.0, 8.0, 7.5)):
    """8 * 4^k triangles: an octahedron's faces cut at edge midpoints, vertices on an ellipsoid."""
    V = [(1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0), (-1.0, 0.0, 0.0), (0.0, -1.0, 0.0), (0.0, 0.0, -1.0)]
    T = [(0, 1, 2), (1, 3, 2), (3, 4, 2), (4, 0, 2), (1, 0, 5), (3, 1, 5), (4, 3, 5), (0, 4, 5)]
    for _ in range(k):
        at, out = {}, []

        def mid(a, b):
            e = (min(a, b), max(a, b))
            if e not in at:
                m = [(V[a][i] + V[b][i]) * 0.5 for i in range(3)]
                r = float(np.sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2]))
                V.append((m[0] / r, m[1] / r, m[2] / r))
                at[e] = len(V) - 1
            return at[e]

        for a, b, c in T:
            ab, bc, ca = mid(a, b), mid(b, c), mid(c, a)
            out += [(a, ab, ca), (ab, b, bc), (ca, bc, c), (ab, bc, ca)]
        T = out
    return np.array(V) * np.array(radii), np.array(T, np.int32)


def vector(n, seed):
    k = np.arange(n, dtype=np.int64)
    return (((k * 7919 + seed * 104729) * (k % 13 + 3)) % 2039).astype(np.float64) / 1019.5 - 1.0


def charges(nc):
    k = np.arange(nc, dtype=np.int64)
    P = np.stack([(k * 37 % 41) / 10.0 - 2.0, (k * 29 % 31) / 8.0 - 2.0, (k * 17 % 23) / 6.0 - 2.0], 1)
    return P, (k * 11 % 19) / 12.0 - 0.75


def digest(t):
    return hashlib.sha256(t.cpu().numpy().tobytes()).hexdigest()[:16]


def _ctx(k, nc, **kw):
    V, T = octasphere(k)
    P, q = charges(nc)
    ctx = pb.pb_create(pb.params(**{**dict(eps_in=1.0, eps_out=80.0, kappa=0.1257, eta0=0.8, leaf_size=48, p=6,
                                           precision=pb.PB_MIXED, precond=pb.PB_PRECOND_BLOCK), **kw}))
    pb.pb_mesh_upload(ctx, V, T, P, q)
    pb.pb_build_tree(ctx)
    return ctx, T.shape[0], q


GOLDEN = {
    "fine": {
        "part1": "14b15b36e5246519",
        "part2": "077fff51f87254ab",
        "part0": "be163715916a032a",
        "multi5": "626d4b8bc57e3dd0",
        "precond": "a05cf5ea9a9da3ed",
        "solution": "375c94652347bcfb",
        "states": "dd5ec944b7c97708",
    },
    "coarse": {
        "part1": "470fc96446c44b0d",
        "part2": "c7725ea6c023f28d",
        "part0": "eee220506af239c2",
        "multi5": "a1f68e5b24bac470",
        "precond": "5addd10c5c48a8be",
        "solution": "b3ea6f9332ad403d",
        "states": "04e3621e453171a1",
    },
    "points": {
        "part1": "f9987210333d9ae4",
        "part2": "c35020473aed1b46",
        "part0": "f9987210333d9ae4",
        "multi5": "d5ab2eed86e6f561",
        "precond": "f5accde0c44a4b1f",
        "solution": "63273ef16c784dcd",
    },
}


def outputs(name):
    """Named digests of one configuration."""
    k, kw = {"fine": (5, {}), "coarse": (4, {"leaf_size": 20, "p": 4, "kappa": 0.3}), "points": (4, {"qr": 2})}[name]
    ctx, nt, q = _ctx(k, 40, **kw)
    try:
        out = {}
        x = torch.from_numpy(vector(2 * nt, 1)).cuda()
        y = torch.empty_like(x)
        for part in (1, 2, 0):
            pb.pb_matvec_part(ctx, x, y, part)
            out[f"part{part}"] = digest(y)
        X = torch.from_numpy(np.stack([vector(2 * nt, s) for s in range(2, 7)])).cuda()
        Y = torch.empty_like(X)
        pb.pb_matvec_multi(ctx, X, Y)
        out["multi5"] = digest(Y)
        pb.pb_precond_apply(ctx, x, y)
        out["precond"] = digest(y)
        y.zero_()
        pb.pb_gmres_solve(ctx, y, tol=1e-6, max_iter=100, restart=50)
        out["solution"] = digest(y)
        if name != "points":
            S = torch.zeros((4, 2 * nt), device="cuda", dtype=torch.float64)
            pb.pb_solve_states(ctx, np.stack([q, -0.5 * q, np.roll(q, 1), np.roll(q, 2)]), S, tol=1e-6, max_iter=100,
                               restart=50, warm=2)
            out["states"] = digest(S)
        return out
    finally:
        pb.pb_destroy(ctx)


@pytest.mark.parametrize("name", ["fine", "coarse", "points"])
def test_products_and_solutions_keep_their_bits(name):
    assert outputs(name) == GOLDEN[name]
