"""Parity of the CUDA path (through the C ABI) with the CPU oracle. Needs a GPU.

Tolerances: integer work (tree order, cluster ranges, lists) bit-exact; FP64 mode within
1e-10 relative L2 of the oracle computing the same algorithm; mixed precision within 2e-5
(FP32 arithmetic with FP64 leaf sums); FMM against the dense Galerkin matvec within 1e-4 at
p = 8 (the required accuracy of the method); energies within 1e-3 relative.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import dense, fmm, kirkwood  # noqa: E402
from paper_2110_13778_gb300 import inputs, pb  # noqa: E402

pytestmark = pytest.mark.gpu

KAP = 0.1257


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2110_13778_gb300 import build

    build.build()
    pb.lib()


def _ctx(mesh, **kw):
    prm = pb.params(**kw)
    ctx = pb.pb_create(prm)
    pb.pb_mesh_upload(ctx, mesh.verts, mesh.tris, mesh.qpos, mesh.q)
    pb.pb_build_tree(ctx)
    return ctx


def _dev(x):
    return torch.tensor(np.asarray(x), device="cuda", dtype=torch.float64)


@pytest.fixture(scope="module")
def sphere3():
    m = inputs.kirkwood_ball(3, 2.0, 5, 1.5, seed=3)
    ph = dense.Phys(1.0, 80.0, KAP, qs=3)
    A = dense.assemble(m.verts, m.tris, ph)
    return m, ph, A


@pytest.mark.parametrize("leaf,eta0", [(16, 0.8), (32, 0.5), (8, 0.7)])
def test_tree_bit_exact(sphere3, leaf, eta0):
    m, ph, A = sphere3
    ctx = _ctx(m, leaf_size=leaf, eta0=eta0)
    try:
        st, order, lb, nc, ni, ic, ii = pb.pb_get_tree(ctx, m.nt)
        tr = fmm.Tree(m.verts, m.tris, leaf_size=leaf, eta0=eta0)
        assert st["levels"] == tr.L
        assert np.array_equal(order, tr.order)
        off = 0
        noff = ioff = 0
        for l in range(tr.L + 1):
            n = tr.nclusters(l)
            assert st["nclusters"][l] == n
            assert np.array_equal(lb[off:off + n], tr.begin[l])
            for c in range(n):
                near = ni[noff:noff + nc[off + c]]
                inter = ii[ioff:ioff + ic[off + c]]
                assert np.array_equal(near, tr.near[l][c]), (l, c)
                assert np.array_equal(inter, tr.inter[l][c]), (l, c)
                noff += nc[off + c]
                ioff += ic[off + c]
            off += n
    finally:
        pb.pb_destroy(ctx)


def test_morton_order_large_and_tied():
    """The stable radix sort of the Morton keys (Section 2.4) on 81920 triangles (320 sort tiles,
    a ragged last scan tile) and on two copies of that surface 2e-4 apart, where most keys tie
    with the key of the element 81920 places later (another sort tile): the order must be the
    keys' order with ties by element index, bit for bit."""
    m = inputs.kirkwood_ball(6, 2.0, 3, 1.5, seed=6)
    V2 = np.vstack([m.verts, m.verts + 2e-4])
    T2 = np.vstack([m.tris, m.tris + len(m.verts)])
    for V, T in ((m.verts, m.tris), (V2, T2)):
        ctx = _ctx(inputs.Mesh(V, T, m.qpos, m.q), leaf_size=64, eta0=0.8, precision=pb.PB_FP64)
        try:
            st, order, *_ = pb.pb_get_tree(ctx, len(T))
        finally:
            pb.pb_destroy(ctx)
        key, _, _ = fmm.morton_keys(fmm.centroids(V, T), V)
        ref = np.lexsort((np.arange(len(T)), key))
        assert np.array_equal(order, ref)
        if len(T) > len(m.tris):
            assert np.count_nonzero(np.diff(key[ref]) == 0) > len(m.tris) // 2  # many ties


def test_all_near_fp64_equals_dense(sphere3):
    m, ph, A = sphere3
    ctx = _ctx(m, leaf_size=16, eta0=1e-6, p=2, precision=pb.PB_FP64)
    try:
        x = inputs.random_density(m.nt, 5)
        y = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
        pb.pb_matvec(ctx, _dev(x), y)
        assert _rel(y.cpu().numpy(), A @ x) < 1e-12
    finally:
        pb.pb_destroy(ctx)


def test_float_float_singular_equals_dense(sphere3):
    # the Sauter-Schwab integrals in float-float reproduce the FP64 oracle's Galerkin matrix
    m, ph, A = sphere3
    ctx = _ctx(m, leaf_size=16, eta0=1e-6, p=2, precision=pb.PB_FP64, singular=pb.PB_SINGULAR_FF)
    try:
        x = inputs.random_density(m.nt, 5)
        y = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
        pb.pb_matvec(ctx, _dev(x), y)
        assert _rel(y.cpu().numpy(), A @ x) < 1e-11
    finally:
        pb.pb_destroy(ctx)


@pytest.mark.parametrize("kappa", [KAP, 2.5])
def test_float_float_singular_matches_fp64_on_molecule(kappa):
    # irregular marching-tetrahedra triangles; kappa = 2.5 takes kappa r past 0.5 (FP64 exp branch)
    from paper_2110_13778_gb300 import molecules

    m = molecules.molecule(40, 4040, 1.0)[0]
    x = _dev(inputs.random_density(m.nt, 6))
    ys = []
    for mode in (pb.PB_SINGULAR_FP64, pb.PB_SINGULAR_FF):
        ctx = _ctx(m, leaf_size=32, eta0=0.7, p=4, kappa=kappa, precision=pb.PB_FP64, singular=mode)
        try:
            y = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
            pb.pb_matvec_part(ctx, x, y, 1)
            ys.append(y.cpu().numpy())
        finally:
            pb.pb_destroy(ctx)
    assert _rel(ys[1], ys[0]) < 1e-11


@pytest.mark.parametrize("p,adaptive", [(4, 0), (6, 0), (8, 0), (3, 1), (5, 0)])
def test_fmm_fp64_matches_oracle_fmm(sphere3, p, adaptive):
    m, ph, A = sphere3
    ctx = _ctx(m, leaf_size=16, eta0=0.8, p=p, adaptive=adaptive, precision=pb.PB_FP64)
    try:
        x = inputs.random_density(m.nt, 9)
        xd = _dev(x)
        y = torch.empty_like(xd)
        pb.pb_matvec(ctx, xd, y)
        tr = fmm.Tree(m.verts, m.tris, leaf_size=16, eta0=0.8)
        yo = fmm.matvec(tr, m.verts, m.tris, x, ph, p, adaptive=bool(adaptive), A=A)
        assert _rel(y.cpu().numpy(), yo) < 1e-10
        # far field alone (no near, no mass)
        yf = torch.empty_like(xd)
        pb.pb_matvec_part(ctx, xd, yf, 2)
        f1, f2 = fmm.far_field(tr, m.verts, m.tris, x, ph, p, adaptive=bool(adaptive))
        assert _rel(yf.cpu().numpy(), np.r_[f1, f2]) < 1e-10
    finally:
        pb.pb_destroy(ctx)


def test_fmm_p8_within_1e4_of_dense(sphere3):
    m, ph, A = sphere3
    for prec in (pb.PB_FP64, pb.PB_MIXED):
        ctx = _ctx(m, leaf_size=16, eta0=0.8, p=8, precision=prec)
        try:
            x = inputs.random_density(m.nt, 11)
            y = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
            pb.pb_matvec(ctx, _dev(x), y)
            assert _rel(y.cpu().numpy(), A @ x) < 1e-4
        finally:
            pb.pb_destroy(ctx)


@pytest.mark.parametrize("p,adaptive", [(4, 0), (6, 0), (8, 0), (10, 0), (5, 0), (3, 1), (2, 0), (7, 0), (9, 0)])
def test_mixed_matches_oracle_fmm(sphere3, p, adaptive):
    # p = 4, 6, 8 run the generated MtL bodies; p = 10, 5, 2, 7, 9 and the adaptive orders
    # (3..6 by level) the generic FP32 recurrence MtL; every order runs its own fixed-order LtP
    m, ph, A = sphere3
    ctx = _ctx(m, leaf_size=16, eta0=0.8, p=p, adaptive=adaptive, precision=pb.PB_MIXED)
    try:
        x = inputs.random_density(m.nt, 13)
        y = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
        pb.pb_matvec(ctx, _dev(x), y)
        tr = fmm.Tree(m.verts, m.tris, leaf_size=16, eta0=0.8)
        yo = fmm.matvec(tr, m.verts, m.tris, x, ph, p, adaptive=bool(adaptive), A=A)
        assert _rel(y.cpu().numpy(), yo) < 2e-5
        yf = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
        pb.pb_matvec_part(ctx, _dev(x), yf, 2)
        f1, f2 = fmm.far_field(tr, m.verts, m.tris, x, ph, p, adaptive=bool(adaptive))
        assert _rel(yf.cpu().numpy(), np.r_[f1, f2]) < 1e-4
    finally:
        pb.pb_destroy(ctx)


def test_rhs_and_energy_match_oracle(sphere3):
    m, ph, A = sphere3
    for prec, tol in ((pb.PB_FP64, 1e-12), (pb.PB_MIXED, 1e-6)):
        ctx = _ctx(m, leaf_size=16, eta0=0.8, p=4, precision=prec)
        try:
            b = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
            pb.pb_rhs(ctx, b)
            bo = dense.rhs(m, ph)
            assert _rel(b.cpu().numpy(), bo) < tol
            x = np.linalg.solve(A, bo)
            E = pb.pb_solvation_energy(ctx, _dev(x))
            Eo = dense.energy(m, ph, x)
            assert abs(E - Eo) < tol * abs(Eo)
        finally:
            pb.pb_destroy(ctx)


def test_block_preconditioner_matches_leaf_blocks(sphere3):
    m, ph, A = sphere3
    ctx = _ctx(m, leaf_size=16, eta0=0.8, p=4, precond=pb.PB_PRECOND_BLOCK)
    try:
        tr = fmm.Tree(m.verts, m.tris, leaf_size=16, eta0=0.8)
        r = inputs.random_density(m.nt, 17)
        z = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
        pb.pb_precond_apply(ctx, _dev(r), z)
        N = m.nt
        zo = np.zeros(2 * N)
        for c in range(tr.nclusters(tr.L)):
            e = tr.order[tr.begin[tr.L][c]:tr.end[tr.L][c]]
            idx = np.r_[e, N + e]
            zo[idx] = np.linalg.solve(A[np.ix_(idx, idx)], r[idx])
        assert _rel(z.cpu().numpy(), zo) < 1e-10
    finally:
        pb.pb_destroy(ctx)


@pytest.mark.parametrize("prec,precond", [(pb.PB_FP64, pb.PB_PRECOND_BLOCK), (pb.PB_MIXED, pb.PB_PRECOND_BLOCK),
                                          (pb.PB_FP64, pb.PB_PRECOND_DIAG), (pb.PB_MIXED, pb.PB_PRECOND_NONE)])
def test_gmres_solution_and_energy(sphere3, prec, precond):
    m, ph, A = sphere3
    ctx = _ctx(m, leaf_size=16, eta0=0.6, p=8, precision=prec, precond=precond)
    try:
        x = torch.zeros(2 * m.nt, device="cuda", dtype=torch.float64)
        tol = 1e-8 if prec == pb.PB_FP64 else 1e-6
        info = pb.pb_gmres_solve(ctx, x, tol=tol, max_iter=200, restart=50)
        assert info.status == pb.PB_OK and info.rel_residual < 1.5 * tol
        xo = np.linalg.solve(A, dense.rhs(m, ph))
        assert _rel(x.cpu().numpy(), xo) < 1e-4
        E = pb.pb_solvation_energy(ctx, x)
        Eo = dense.energy(m, ph, xo)
        assert abs(E - Eo) < 1e-4 * abs(Eo)
    finally:
        pb.pb_destroy(ctx)


def test_kirkwood_small_sphere_energy():
    # the 2 A, +1 e Kirkwood sphere at 1280 triangles: oracle parity and the closed form
    m = inputs.kirkwood_centered(3, 2.0, 1.0)
    ph = dense.Phys(1.0, 80.0, KAP, qs=3)
    xo, A, b = dense.solve(m, ph)
    Eo = dense.energy(m, ph, xo)
    ex = kirkwood.centered(1.0, 2.0, 1.0, 80.0, KAP)
    for prec in (pb.PB_FP64, pb.PB_MIXED):
        ctx = _ctx(m, leaf_size=16, eta0=0.8, p=8, precision=prec)
        try:
            x = torch.zeros(2 * m.nt, device="cuda", dtype=torch.float64)
            info = pb.pb_gmres_solve(ctx, x, tol=1e-6, max_iter=100, restart=50)
            assert info.status == pb.PB_OK
            E = pb.pb_solvation_energy(ctx, x)
            assert abs(E - Eo) < 1e-3 * abs(Eo)
            assert abs(E - ex) < 0.015 * abs(ex)
        finally:
            pb.pb_destroy(ctx)


def test_bad_mesh_rejected():
    V, T = inputs.icosphere(1, 1.0)
    prm = pb.params()
    ctx = pb.pb_create(prm)
    try:
        Tb = T.copy()
        Tb[3, 1] = 10_000
        with pytest.raises(pb.PBError) as e:
            pb.pb_mesh_upload(ctx, V, Tb, np.zeros((1, 3)), np.ones(1))
        assert e.value.code == pb.PB_ERR_MESH
        Tz = T.copy()
        Tz[0] = [0, 0, 1]
        with pytest.raises(pb.PBError):
            pb.pb_mesh_upload(ctx, V, Tz, np.zeros((1, 3)), np.ones(1))
        with pytest.raises(pb.PBError) as e:
            pb.pb_build_tree(ctx)
        assert e.value.code == pb.PB_ERR_STATE
    finally:
        pb.pb_destroy(ctx)


def test_tiny_and_ragged_meshes():
    # single-level tree (everything near) and a mesh smaller than one leaf
    for lev, leaf in ((0, 64), (1, 64), (2, 7)):
        V, T = inputs.perturbed_sphere(lev, 3.0, 0.1, seed=lev) if lev else inputs.icosphere(0, 3.0)
        m = inputs.Mesh(V, T, np.zeros((1, 3)), np.ones(1))
        ph = dense.Phys(1.0, 80.0, KAP, qs=3)
        A = dense.assemble(V, T, ph)
        ctx = _ctx(m, leaf_size=leaf, eta0=0.8, p=6, precision=pb.PB_FP64)
        try:
            x = inputs.random_density(m.nt, 2)
            y = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
            pb.pb_matvec(ctx, _dev(x), y)
            tr = fmm.Tree(V, T, leaf_size=leaf, eta0=0.8)
            yo = fmm.matvec(tr, V, T, x, ph, 6, A=A)
            assert _rel(y.cpu().numpy(), yo) < 1e-10
        finally:
            pb.pb_destroy(ctx)


@pytest.mark.parametrize("leaf,levels", [(1000, 1), (1, 3), (3, 2), (40, 0), (70, 0)])
@pytest.mark.parametrize("part", [0, 1])
def test_fp64_pair_tiles_ragged_leaves(leaf, levels, part):
    # chunks of 1 to 32 elements: leaves of one and a few elements, remainders on both sides of a
    # tile, one leaf of many chunks; bar as above (FP64 mode within 1e-10 of the oracle FMM)
    V, T = inputs.perturbed_sphere(3, 2.0, 0.2, seed=17)
    T = T[:1277] if levels == 0 else T
    m = inputs.Mesh(V, T, np.zeros((1, 3)), np.ones(1))
    ctx = _ctx(m, eta0=0.8, leaf_size=leaf, levels=levels, p=6, precision=pb.PB_FP64, precond=pb.PB_PRECOND_DIAG)
    try:
        tr = fmm.Tree(V, T, leaf_size=leaf, eta0=0.8, levels=levels) if levels else fmm.Tree(V, T, leaf_size=leaf, eta0=0.8)
        x = inputs.random_density(m.nt, leaf)
        y = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
        pb.pb_matvec_part(ctx, _dev(x), y, part)
        if part == 0:
            ph = dense.Phys(1.0, 80.0, KAP, qs=3)
            assert _rel(y.cpu().numpy(), fmm.matvec(tr, V, T, x, ph, 6)) < 1e-10
        z = torch.empty_like(y)
        pb.pb_matvec_part(ctx, _dev(x), z, part)
        assert torch.equal(y, z)  # no atomics: the same product twice is the same bits
    finally:
        pb.pb_destroy(ctx)


@pytest.mark.parametrize("kappa", [0.0, 0.02, KAP, 0.6, 3.0])
@pytest.mark.parametrize("leaf,qr", [(1000, 0), (5, 0), (45, 0), (20, 2)])
def test_mixed_near_tiles_against_fp64(kappa, leaf, qr):
    # tiles within, across and beyond kappa r = 0.125 (where the screening series ends), full and
    # remainder chunks on either side, points of a rule. Both runs hold the same FP64 corrections
    # and mass terms, so what is left is the FP32 pair terms: about ten roundings of 6e-8 each
    V, T = inputs.perturbed_sphere(3, 2.0, 0.2, seed=23)
    m = inputs.Mesh(V, T[:1271], np.zeros((1, 3)), np.ones(1))
    x = _dev(inputs.random_density(m.nt, 5))
    got = []
    for prec in (pb.PB_FP64, pb.PB_MIXED):
        ctx = _ctx(m, kappa=kappa, eta0=0.8, leaf_size=leaf, p=4, qr=qr, precision=prec, precond=pb.PB_PRECOND_DIAG,
                   singular=pb.PB_SINGULAR_FP64)
        try:
            y = torch.empty_like(x)
            pb.pb_matvec_part(ctx, x, y, 1)
            got.append(y.cpu().numpy())
        finally:
            pb.pb_destroy(ctx)
    assert _rel(got[1], got[0]) < 6e-7


@pytest.mark.parametrize("n", [1023, 1024, 16383, 16384, 16385, 16384 + 1024])
def test_scans_across_one_block_and_tiles(n):
    # the build's scans at the edges of the one-block form (16384 values) and of the tiles behind it:
    # the order, the cluster ranges and the touching counts of a mesh of n triangles
    V, T = inputs.icosphere(5 if n > 5120 else 4, 3.0)
    T = T[:n]
    m = inputs.Mesh(V, T, np.zeros((1, 3)), np.ones(1))
    ctx = _ctx(m, leaf_size=24, eta0=0.8, p=2, precision=pb.PB_MIXED, precond=pb.PB_PRECOND_DIAG)
    try:
        st, order, lb, nc, ni, ic, ii = pb.pb_get_tree(ctx, m.nt)
        tr = fmm.Tree(V, T, leaf_size=24, eta0=0.8)
        assert np.array_equal(order, tr.order)
        assert np.array_equal(lb[-len(tr.begin[tr.L]):], tr.begin[tr.L])
        share = {}
        for t in T:
            for v in t:
                share[v] = share.get(v, 0) + 1
        # touching ordered pairs: by vertex, minus those counted twice or three times (shared edges, i == j)
        E = np.sort(T[:, [0, 1, 1, 2, 2, 0]].reshape(-1, 2), 1)
        _, k = np.unique(E, axis=0, return_counts=True)
        assert st["touching"] == sum(c * c for c in share.values()) - int((k * k).sum()) + m.nt
    finally:
        pb.pb_destroy(ctx)


@pytest.mark.parametrize("nc", [1, 255, 257, 512, 513, 1025, 2100])
def test_rhs_charge_groups(sphere3, nc):
    # tiles of 256 charges, one group of threads up to 512 charges and four beyond, with empty and ragged
    # last tiles. Charges of one sign inside a sphere: all terms of either half have one sign, so the
    # FP32 sum of a tile (256 terms) is within 256 * 2^-24 = 1.5e-5 of itself
    m, ph, _ = sphere3
    rng = np.random.default_rng(nc)
    R = float(np.linalg.norm(m.verts[0]))
    m = inputs.Mesh(m.verts, m.tris, rng.uniform(-0.4, 0.4, (nc, 3)) * R, rng.uniform(0.1, 1.0, nc))
    ctx = _ctx(m, leaf_size=48, p=4, precision=pb.PB_MIXED)
    try:
        b = torch.empty(2 * m.nt, device="cuda", dtype=torch.float64)
        pb.pb_rhs(ctx, b)
        np.testing.assert_allclose(b.cpu().numpy(), dense.rhs(m, ph), rtol=2e-5)
    finally:
        pb.pb_destroy(ctx)


def test_fp64_near_field_of_a_large_leaf_in_bounded_memory():
    # one leaf of 81,920 elements: 3.3 million pair tiles, whose sums (1 KB each) are held for 262,144 tiles at
    # a time, 256 MB beside 0.1 GB of lists and records; a few rows against the direct sum in FP64.
    # Bar as above (1e-10)
    V, T = inputs.icosphere(6, 30.0)
    m = inputs.Mesh(V, T, np.zeros((1, 3)), np.ones(1))
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    ctx = _ctx(m, eta0=0.8, leaf_size=10**6, p=2, qs=2, precision=pb.PB_FP64, precond=pb.PB_PRECOND_DIAG)
    try:
        assert pb.pb_get_tree_stats(ctx)["max_leaf"] == m.nt
        assert free0 - torch.cuda.mem_get_info()[0] < 1 << 30
        x = _dev(inputs.random_density(m.nt, 3))
        y, z = torch.empty_like(x), torch.empty_like(x)
        pb.pb_matvec_part(ctx, x, y, 1)
        # rows of elements that touch nothing in the density's support, against the sum over it
        P = _dev(V[T].mean(1))
        E1, E2 = _dev(V[T[:, 1]] - V[T[:, 0]]), _dev(V[T[:, 2]] - V[T[:, 0]])
        N = torch.linalg.cross(E1, E2)
        A = N.norm(dim=1) / 2
        N = N / (2 * A[:, None])
        far = P[:, 2] > 0
        xs = x.view(2, -1) * far  # support: the upper half
        pb.pb_matvec_part(ctx, xs.reshape(-1).contiguous(), z, 1)
        rows = torch.nonzero(P[:, 2] < -1.0).ravel()[:: m.nt // 97]
        d = P[rows, None, :] - P[None]
        r2 = (d * d).sum(-1)
        r = r2.sqrt()
        t = KAP * r
        e = torch.exp(-t)
        xd, yd = (N[rows, None] * d).sum(-1), (N[None] * d).sum(-1)
        nn = N[rows] @ N.T
        ph, dph = (A * xs[0])[None], (A * xs[1])[None]
        g3 = 1 / r**3
        k1, k2 = -torch.expm1(-t) / r, yd * g3 * (80.0 * e * (1 + t) - 1)
        k3 = -xd * g3 * (1 - e * (1 + t) / 80.0)
        k4 = g3 * ((3 - e * (3 + 3 * t + t * t)) * xd * yd / r2 - (1 - e * (1 + t)) * nn)
        on = far[None]
        s1 = torch.where(on, k1 * dph + k2 * ph, 0.0).sum(1) / (4 * np.pi)
        s2 = torch.where(on, k3 * dph + k4 * ph, 0.0).sum(1) / (4 * np.pi)
        want = torch.stack([-A[rows] * s1, -A[rows] * s2])
        assert _rel(z.view(2, -1)[:, rows].cpu().numpy(), want.cpu().numpy()) < 1e-10
        # linear: the product of both halves' densities adds up
        pb.pb_matvec_part(ctx, (x.view(2, -1) * ~far).reshape(-1).contiguous(), xs.view(-1), 1)
        assert _rel((xs.view(-1) + z).cpu().numpy(), y.cpu().numpy()) < 1e-12
    finally:
        pb.pb_destroy(ctx)


def test_several_vectors_add_tiles_in_fp64():
    # 248 elements in one leaf: every row's eight tiles are one work item, summed in FP64. Densities u
    # on the first chunk and w = 2^-k on the third are evaluated alone and together, so that the rows of a
    # third place are sums of the same two FP32 tile sums: y(u + w) = y(u) + y(w) up to five roundings, of
    # the sum, of the three rows and of the addition below, each 2^-53 of the largest value
    V, T = inputs.icosphere(3, 4.0)
    T = T[:248]
    m = inputs.Mesh(V, T, np.zeros((1, 3)), np.ones(1))
    ctx = _ctx(m, eta0=0.8, leaf_size=1000, p=2, precision=pb.PB_MIXED, precond=pb.PB_PRECOND_DIAG)
    try:
        order = pb.pb_get_tree(ctx, m.nt)[1]
        u, w = np.zeros(m.nt), np.zeros(m.nt)
        u[order[:32]] = inputs.random_density(m.nt, 1)[:32]
        w[order[64:96]] = inputs.random_density(m.nt, 2)[:32]
        near = np.isin(T, T[np.concatenate([order[:32], order[64:96]])]).any(1)  # the corrections' rows
        rows = np.tile(~near, 2)
        assert rows.sum() > 150
        X = []
        for k in (8, 16, 20, 24, 28):
            for a, b in ((u, 0 * w), (0 * u, w * 2.0**-k), (u, w * 2.0**-k)):
                X.append(np.concatenate([a + b, 0.5 * a - b]))
        X = _dev(np.stack(X + [X[0]]))
        Y = torch.empty_like(X)
        pb.pb_matvec_multi(ctx, X, Y)
        Y = Y.cpu().numpy()[:, rows]
        for a, b, c in zip(Y[0:15:3], Y[1:15:3], Y[2:15:3]):
            big = np.maximum(np.maximum(np.abs(a), np.abs(b)), np.abs(c))
            assert np.all(np.abs(c - (a + b)) <= 5 * 2.0**-53 * big)
    finally:
        pb.pb_destroy(ctx)


def test_scans_of_more_than_4096_tiles():
    # 1,440,000 elements: the scan over three counts per element takes 4219 tiles, whose sums are scanned by
    # themselves. It places the unordered touching pairs of the float-float integrals; the FP64 integrals
    # do without, and both forms agree to 1e-11 (the bar of the float-float integrals)
    n, w = 1200, 600
    u, v = np.meshgrid(np.arange(n) * (2 * np.pi / n), np.arange(w) * (2 * np.pi / w), indexing="ij")
    V = np.stack([(60 + 25 * np.cos(v)) * np.cos(u), (60 + 25 * np.cos(v)) * np.sin(u), 25 * np.sin(v)], -1).reshape(-1, 3)
    i, j = np.meshgrid(np.arange(n), np.arange(w), indexing="ij")
    a, b = (i * w + j).ravel(), (((i + 1) % n) * w + j).ravel()
    c, d = (((i + 1) % n) * w + (j + 1) % w).ravel(), (i * w + (j + 1) % w).ravel()
    T = np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, d], 1)]).astype(np.int32)
    m = inputs.Mesh(V, T, np.zeros((1, 3)), np.ones(1))
    x = _dev(inputs.random_density(m.nt, 7))
    got = []
    for singular in (pb.PB_SINGULAR_FF, pb.PB_SINGULAR_FP64):
        ctx = _ctx(m, eta0=0.8, leaf_size=24, p=2, qs=2, precision=pb.PB_MIXED, precond=pb.PB_PRECOND_DIAG, singular=singular)
        try:
            assert pb.pb_get_tree_stats(ctx)["touching"] == 13 * m.nt  # six triangles at every vertex
            y = torch.empty_like(x)
            pb.pb_matvec_part(ctx, x, y, 1)
            got.append(y.cpu().numpy())
        finally:
            pb.pb_destroy(ctx)
    assert _rel(got[0], got[1]) < 1e-11


@pytest.mark.parametrize("p", [9, 10])
@pytest.mark.parametrize("prec,tol", [(pb.PB_FP64, 1e-13), (pb.PB_MIXED, 1e-6)])
def test_several_vectors_at_high_orders(p, prec, tol):
    # orders above 8 have more multi-indices than threads in the leaf moments: several vectors take the
    # one-vector form of that kernel. Bars: the roundings of the working precision
    V, T = inputs.perturbed_sphere(4, 9.0, 0.2, seed=5)
    m = inputs.Mesh(V, T, np.zeros((1, 3)), np.ones(1))
    ctx = _ctx(m, eta0=0.8, leaf_size=16, p=p, precision=prec, precond=pb.PB_PRECOND_DIAG)
    try:
        X = _dev(np.stack([inputs.random_density(m.nt, s) for s in range(5)]))
        Y, y = torch.empty_like(X), torch.empty_like(X[0])
        pb.pb_matvec_multi(ctx, X, Y)
        for r in range(5):
            pb.pb_matvec_part(ctx, X[r].contiguous(), y, 0)
            assert _rel(Y[r].cpu().numpy(), y.cpu().numpy()) < tol
    finally:
        pb.pb_destroy(ctx)
