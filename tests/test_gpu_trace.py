"""Cells by edge tracing (csrc/trace_impl.cuh) at the sizes where they can go
wrong: lists that hold every other generator, lists shorter and longer than the
planes of a group, cells with more vertices than its slots, cells that every
round leaves open, degenerate vertices (the certificate refuses them), point
counts that leave groups and blocks partly empty, and small sets in a batch.
Calls of up to 12,288 points build every cell by a warp ("warps"); the same
points in a batch beside enough others go through the groups of 8 lanes, the
walk of their open cells and the warps for what these leave ("groups").
Both forms against the FP64 oracle, to the tolerances of the other parity tests
(FP32: 1e-5 relative, about 150 roundings of the volume's terms, neighbours but
for faces below 1e-6 V^(2/3); FP64: 1e-12, the oracle's own bound on cells of
clumps, neighbours exact)."""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2412_04514_gb300 as vt
from geometry_match import emitted_cell, match_cell, oracle_cell
from paper_2412_04514_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "fp64": 1e-12}
GEO = ("vtx_off", "vtx", "face_off", "face_nbr", "face_vtx_off", "face_vtx")
ROUTES = pytest.mark.parametrize("route", ["warps", "groups"])
PRECS = pytest.mark.parametrize("prec", ["fp32", "fp64"])


def run(pts, prec, route, emit, **kw):
    """The cells of ``pts`` as numpy arrays: of a call of their own, or of a
    batch whose second set makes it large enough for the groups."""
    p = vt.Params(precision=prec, emit=emit, **kw)
    n = len(pts)
    if route == "warps":
        c = vt.tessellate(torch.from_numpy(pts).cuda(), p)
    else:
        both = np.concatenate([pts, W.uniform(12_301, 77)])
        c = vt.tessellate_batch(torch.from_numpy(both).cuda(), [0, n, len(both)], p)
        assert c.stats["clip_launches"] >= 4  # two rounds of groups, the warps, the clipper
    assert c.stats["status"] == "VT_OK"
    out = {}
    for name in ("vol", "cen", "nbr_off", "nbr") + GEO:
        t = getattr(c, name)
        if t is not None:
            out[name] = t.cpu().numpy()
    out["vol"], out["cen"] = out["vol"][:n], out["cen"][:n]
    if "nbr" in out:
        out["nbr_off"] = out["nbr_off"][:n + 1]
        out["nbr"] = out["nbr"][:out["nbr_off"][-1]]
    return out


def least_det(V, faces):
    """The smallest |det| of three faces' unit normals over the vertices of a cell (1e-7 at least)."""
    normal = []
    for _, loop in faces:
        P = V[loop] - V[loop[0]]
        a = np.cross(P[1:-1], P[2:]).sum(0)
        normal.append(a / max(np.linalg.norm(a), 1e-300))
    at = [[normal[f] for f, (_, loop) in enumerate(faces) if k in loop] for k in range(len(V))]
    return max(1e-7, min(abs(np.linalg.det(np.stack(n[:3]))) for n in at if len(n) >= 3))


def check(pts, prec, route="warps", periodic=False, generic=True, **kw):
    want = oracle.tessellate(pts, periodic=periodic, geometry=generic)
    n = len(pts)
    c = run(pts, prec, route, ("nbr", "vol", "cen") + (("geom",) if generic else ()), periodic=periodic, **kw)
    np.testing.assert_allclose(c["vol"], want["vol"], rtol=TOL[prec])
    np.testing.assert_allclose(c["cen"], want["cen"], rtol=TOL[prec], atol=TOL[prec] * 1e-2)
    if not generic:
        return
    differ = set()
    if prec == "fp64":
        assert np.array_equal(c["nbr_off"], want["nbr_off"]) and np.array_equal(c["nbr"], want["nbr"])
    else:
        for i in range(n):
            got, ref = (sorted(x["nbr"][x["nbr_off"][i]:x["nbr_off"][i + 1]].tolist()) for x in (c, want))
            if got == ref:
                continue
            differ.add(i)
            faces = slice(want["face_off"][i], want["face_off"][i + 1])
            for j in set(got) ^ set(ref):
                areas = want["face_area"][faces][want["face_tag"][faces] == j]
                assert len(areas) == 0 or areas.min() < 1e-6 * want["vol"][i] ** (2 / 3), (i, j, areas)
        assert len(differ) <= max(2, 1e-3 * n)
    # every cell is a simple polyhedron: V = 2 F - 4, three faces at each vertex
    v, f = np.diff(c["vtx_off"])[:n], np.diff(c["face_off"])[:n]
    assert np.array_equal(v, 2 * f - 4)
    deg = np.diff(c["face_vtx_off"])[:c["face_off"][n]]
    assert deg.min() >= 3 and deg.sum() == 3 * v.sum()
    # vertices and loops of some cells, matched one to one
    geo = [c[g] for g in GEO]
    for i in range(0, n, max(1, n // 40)):
        if i in differ:
            continue
        V, faces = emitted_cell(geo, i)
        Wv, wfaces = oracle_cell(want, i)
        amax = max(1.0, np.abs(Wv).max())
        # (Cramer's rule leaves 32 roundings / |det| of a vertex's distance from the generator)
        atol = 32 * 2.0 ** -53 / least_det(Wv, wfaces) * np.linalg.norm(Wv - pts[i], axis=1).max() + 1e-15 * amax
        if prec == "fp32":
            atol += 1e-5 * np.cbrt(want["vol"][i]) + 4 * np.finfo(np.float32).eps * amax
        match_cell(V, faces, Wv, wfaces, atol)


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("make", [lambda: W.uniform(2, 1), lambda: W.uniform(20, 2), lambda: W.uniform(33, 3),
                                  lambda: W.uniform(34, 4), lambda: W.uniform(4001, 5),
                                  lambda: W.mixed(4001, 6, n_clumps=3),
                                  lambda: np.concatenate([W.uniform(50, 7), np.random.default_rng(8).normal(
                                      0.5, 1e-2, (4000, 3)).astype(np.float32)])],
                         ids=["2", "20", "33", "34", "uniform", "clumps", "sparse beside a clump"])
def test_lists_hold_every_generator_below_their_reach(make, periodic):
    # the lists as the call leaves them in its workspace: found by the nearest
    # generators, which come first, and followed by the reaches
    pts = make()
    n, k = len(pts), 32
    p = vt.Params(precision="fp32", emit=("vol",), periodic=periodic)
    ws = vt.Workspace(p, n)
    ws.buf.zero_()
    c = vt.tessellate(torch.from_numpy(pts).cuda(), p, workspace=ws, want_perm=True)
    assert c.stats["knn_queries"] == n  # (the clipper's lists would lie in the same place)
    x = pts[c.perm.cpu().numpy()[:n]].astype(np.float64)
    off = x[None] - x[:, None]
    if periodic:  # (the nearest image stands for the others: they are farther than half a period)
        off -= np.rint(off)
    d2 = (off ** 2).sum(-1)
    np.fill_diagonal(d2, np.inf)
    buf = ws.buf[:ws.buf.numel() // 4 * 4].view(torch.int32).cpu().numpy()
    mask = (1 << 24) - 1 if periodic else -1
    rows = np.arange(min(n, 16))
    near = d2[rows].min(1)
    at = np.arange(0, len(buf) - n * k, 64)
    for r in rows:
        first = buf[at + k * r] & mask
        ok = (buf[at + k * r] >= 0) & (first < n)
        at = at[ok][np.isclose(d2[r, first[ok]], near[r], rtol=1e-5, atol=0)]
        row = buf[at[:, None] + k * r + np.arange(k)]
        at = at[((row == -1) | ((row >= 0) & ((row & mask) < n))).all(1) & (row[:, 1:] != 0).any(1)]
    assert len(at) == 1, at
    lists = buf[at[0]:at[0] + n * k].reshape(n, k)
    size = max(n * k, 64 * 32)
    reach = buf[at[0] + (size + 63) // 64 * 64:][:n].view(np.float32).astype(np.float64)
    for i in range(n):
        ids = lists[i][lists[i] != -1]
        if periodic:
            code = ids >> 24
            t = np.stack([code // 25 - 2, code // 5 % 5 - 2, code % 5 - 2], 1)
            key = ((x[ids & mask] + t - x[i]) ** 2).sum(1)
        else:
            key = d2[i, ids]
        assert len(set(ids.tolist())) == len(ids) and i not in (ids & mask)
        assert key[0] <= key.min() * (1 + 1e-5) and (key < reach[i] * (1 + 1e-5)).all()
        below = np.flatnonzero(d2[i] < min(reach[i], 0.25 if periodic else np.inf) * (1 - 1e-5))
        assert set(below.tolist()) <= set((ids & mask).tolist()), i
        if not periodic:
            assert (reach[i] > 1e30) == (len(ids) == n - 1)


@ROUTES
@PRECS
@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 32, 33, 34, 35, 63, 65, 127, 129, 515])
def test_small_counts(n, prec, route):
    check(W.uniform(n, 100 + n), prec, route)


@ROUTES
@PRECS
@pytest.mark.parametrize("k0,k_max", [(6, 12), (12, 12), (16, 31), (17, 34), (17, 40), (18, 36), (40, 70), (64, 64)])
def test_list_lengths(k0, k_max, prec, route):
    check(W.mixed(3001, 5, n_clumps=3), prec, route, k0=k0, k_max=k_max)


@ROUTES
@PRECS
@pytest.mark.parametrize("n", [40, 300, 1201])
def test_periodic(n, prec, route):
    check(W.mixed(n, 9, n_clumps=2, periodic=True), prec, route, periodic=True)


@ROUTES
@PRECS
@pytest.mark.parametrize("around", [20, 26, 27, 40, 60])
def test_many_faced_cells(around, prec, route):
    # a generator inside a shell of `around` others at about one distance: its
    # cell has up to around faces (26 fill the vertex slots of a group)
    rng = np.random.default_rng(around)
    d = rng.standard_normal((around, 3))
    shell = 0.5 + (0.2 + 1e-3 * rng.random((around, 1))) * d / np.linalg.norm(d, axis=1, keepdims=True)
    far = rng.random((400, 3))
    far = far[np.linalg.norm(far - 0.5, axis=1) > 0.4]
    check(np.concatenate([[[0.5, 0.5, 0.5]], shell, far]).astype(np.float32), prec, route)


@PRECS
@pytest.mark.parametrize("m,move", [(25, 1e-3), (25, 1e-4), (25, 1e-5), (12, 1e-4)])
def test_lattices_that_moved_little(m, move, prec):
    # most cells have planes within float32 round-off of their vertices. Where
    # they are many, the clipper builds them and not the FP64 rays
    rng = np.random.default_rng(m)
    x = (W.cubic_lattice(m) + rng.uniform(-move / m, move / m, (m ** 3, 3))).astype(np.float32)
    want = oracle.tessellate(x)
    for kw in ({}, {"fused": True}):
        cells = vt.tessellate(torch.from_numpy(x).cuda(), vt.Params(precision=prec, emit=("nbr", "vol", "cen"), **kw))
        np.testing.assert_allclose(cells.vol.cpu().numpy(), want["vol"], rtol=TOL[prec])
        np.testing.assert_allclose(cells.cen.cpu().numpy(), want["cen"], rtol=TOL[prec])
        if prec == "fp64":
            assert np.array_equal(cells.nbr_off.cpu().numpy(), want["nbr_off"])
            assert np.array_equal(cells.nbr.cpu().numpy(), want["nbr"])
        elif m == 25:
            assert cells.stats["precision_retries"] < len(x) // 16


@PRECS
@pytest.mark.parametrize("seed", [25, 33, 37])
def test_filaments_validate(seed, prec):
    # points along segments: far cells whose thousands of cutting generators take
    # tens of turns, more than the clipper's slots hold on the way
    rng = np.random.default_rng(seed)
    a, b = 0.1 + 0.8 * rng.random((20, 3)), 0.1 + 0.8 * rng.random((20, 3))
    x = a[:, None] + (b - a)[:, None] * np.linspace(0, 1, 200)[None, :, None] + 3e-3 * rng.standard_normal((20, 200, 3))
    x = np.unique(x.reshape(-1, 3).astype(np.float32), axis=0)
    c = vt.tessellate(torch.from_numpy(x).cuda(), vt.Params(precision=prec, emit=("vol",), periodic=True))
    assert c.stats["status"] == "VT_OK"
    assert abs(float(c.vol.sum()) - 1.0) < TOL[prec]


def test_rays_that_meet_two_planes_within_float_rounding():
    # of so many cells with nearly coincident vertices none may be left to the
    # clipper for an order of two planes along a ray that float32 cannot tell
    rng = np.random.default_rng(0)
    x = (W.cubic_lattice(50) + rng.uniform(-2e-5, 2e-5, (125_000, 3))).astype(np.float32)
    s = vt.tessellate(torch.from_numpy(x).cuda(), vt.Params(precision="fp64", emit=("vol",))).stats
    assert s["knn_queries"] == len(x), s  # (the clipper's cells ask for lists of their own)


def test_sums_of_many_edges():
    # the FP32 form's moments of cells of up to 60 faces (22 edges to a lane) are
    # no further off than the clipper's (k_max = 4 k0 is not traced), whose lanes
    # add at most six terms in float32: root mean squares over 96 cells, which
    # differ by 3% from one set of 96 to another
    err = {True: [], False: []}
    for seed in range(96):
        rng = np.random.default_rng(seed)
        d = rng.standard_normal((60, 3))
        shell = 0.5 + (0.2 + 1e-3 * rng.random((60, 1))) * d / np.linalg.norm(d, axis=1, keepdims=True)
        far = rng.random((200, 3))
        far = far[np.linalg.norm(far - 0.5, axis=1) > 0.4]
        x = torch.from_numpy(np.concatenate([[[0.5, 0.5, 0.5]], shell, far]).astype(np.float32)).cuda()
        want = vt.tessellate(x, vt.Params(precision="fp64", emit=("vol", "m2")))
        for traced in (True, False):
            kw = {} if traced else {"k0": 6, "k_max": 24}
            c = vt.tessellate(x, vt.Params(precision="fp32", emit=("vol", "m2"), **kw))
            err[traced].append([float(c.vol[0] / want.vol[0]) - 1, float(c.m2[0] / want.m2[0]) - 1])
    rms = {k: np.sqrt(np.mean(np.square(v), axis=0)) for k, v in err.items()}
    assert (rms[True] < 1.03 * rms[False]).all(), rms


@ROUTES
@PRECS
def test_sparse_cells_beside_a_dense_clump(prec, route):
    # the lists of the sparse points end inside the clump; thousands of its
    # points lie within twice their radius and the rounds cut them back
    rng = np.random.default_rng(4)
    clump = 0.5 + 2e-3 * rng.standard_normal((6000, 3))
    check(np.concatenate([clump, rng.random((60, 3))]).astype(np.float32), prec, route)


@ROUTES
@PRECS
@pytest.mark.parametrize("make", [lambda: W.cubic_lattice(8), lambda: W.bcc_lattice(6)], ids=["cubic", "bcc"])
def test_lattices(make, prec, route):
    # every vertex of the cubic lattice and the walls' of the BCC lattice have
    # more than three planes: the certificate sends the cells to the clipper
    check(make(), prec, route, generic=False)


@ROUTES
@PRECS
def test_more_equal_distances_than_a_list_holds(prec, route):
    # 48 generators at one exact distance around the middle one: no limit keeps
    # between a list's length less one and a list's length of them. (Nothing
    # else: the middle cell's vertices have up to eight planes, and beside
    # generic points no schedule validates such a cell.)
    d = np.array([1.0, 2.0, 4.0]) / 32
    ring = [0.5 + np.array(s) * d[list(o)] for o in itertools.permutations(range(3))
            for s in itertools.product([-1, 1], repeat=3)]
    pts = np.concatenate([[[0.5, 0.5, 0.5]], ring]).astype(np.float32)
    check(pts, prec, route, generic=False)


@PRECS
@pytest.mark.parametrize("n", [3, 20, 300])
def test_box_whose_plane_products_overflow(n, prec):
    # a box of 2^40: the float32 products of a vertex's three planes overflow,
    # its error bound can become infinite, and short lists have padding planes.
    # The cells are those of the unit box, scaled by a power of two.
    pts = W.uniform(n, 60 + n)
    want = oracle.tessellate(pts)
    scale = 2.0 ** 40
    cells = vt.tessellate(torch.from_numpy(pts * np.float32(scale)).cuda(),
                          vt.Params(precision=prec, emit=("nbr", "vol", "cen"), box_hi=(scale,) * 3))
    np.testing.assert_allclose(cells.vol.cpu().numpy() / scale ** 3, want["vol"], rtol=TOL[prec])
    if prec == "fp64":  # (first moments, fourth powers of a length, overflow float32 here)
        np.testing.assert_allclose(cells.cen.cpu().numpy() / scale, want["cen"], rtol=1e-12)


@pytest.mark.parametrize("n,clumps,k", [(300, 0, -33), (2000, 2, -26), (20_000, 10, -26)])
def test_small_scales(n, clumps, k):
    # the clouds' products of three normals (and of their squares) underflow float32
    pts = W.mixed(n, 3, n_clumps=clumps) if clumps else W.uniform(n, 1)
    want = oracle.tessellate(pts)
    scale = 2.0 ** k
    cells = vt.tessellate(torch.from_numpy(pts * np.float32(scale)).cuda(),
                          vt.Params(precision="fp32", emit=("nbr", "vol"), box_hi=(scale,) * 3))
    np.testing.assert_allclose(cells.vol.cpu().numpy() / scale ** 3, want["vol"], rtol=TOL["fp32"])


@PRECS
@pytest.mark.parametrize("spacing", [1e-20, 1e-19, 1e-18, 1e-13])
def test_generators_whose_squares_underflow(spacing, prec):
    # three generators on a line: the cell between two others is a slab of the
    # box as thick as their spacing. Beyond the range of the certificate's bounds
    # the cells are the clipper's (k_max = 4 k0 is not traced), whose FP64 form
    # takes a plane within 1e-14 R of the vertices it cuts as touching them.
    x = np.array([1, 2, 3]) * spacing
    pts = np.stack([x, np.full(3, 0.5), np.full(3, 0.5)], 1).astype(np.float32)
    cells, clip = (vt.tessellate(torch.from_numpy(pts).cuda(), vt.Params(precision=prec, emit=("nbr", "vol"), **kw))
                   for kw in ({}, {"k0": 6, "k_max": 24}))
    torch.testing.assert_close(cells.vol, clip.vol, rtol=TOL[prec], atol=0)
    assert torch.equal(cells.nbr_off, clip.nbr_off) and torch.equal(cells.nbr, clip.nbr)
    if prec == "fp32" or spacing > 1e-14:
        x = pts[:, 0].astype(np.float64)
        cut = [0.0, (x[0] + x[1]) / 2, (x[1] + x[2]) / 2, 1.0]
        np.testing.assert_allclose(cells.vol.cpu().numpy(), np.diff(cut), rtol=TOL[prec])
        assert cells.nbr_off.tolist() == [0, 1, 3, 4] and cells.nbr.tolist() == [1, 0, 2, 1]


def test_box_beyond_float_squares():
    # 2^60: not traced, the clipper's FP64 form builds the unit box's cells scaled
    pts = W.uniform(300, 8)
    want = oracle.tessellate(pts)
    for fused in (False, True):
        cells = vt.tessellate(torch.from_numpy(pts * np.float32(2.0 ** 60)).cuda(),
                              vt.Params(precision="fp64", emit=("nbr", "vol"), box_hi=(2.0 ** 60,) * 3, fused=fused))
        np.testing.assert_allclose(cells.vol.cpu().numpy() / 2.0 ** 180, want["vol"], rtol=1e-12)
        assert np.array_equal(cells.nbr.cpu().numpy(), want["nbr"])


@ROUTES
@PRECS
def test_batch_of_small_sets(prec, route):
    sizes = [1, 2, 0, 7, 33, 34, 35, 200, 1, 1500] + [11_001] * (route == "groups")
    parts = [W.uniform(n, 40 + i) for i, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)])
    b = vt.Batch(torch.from_numpy(np.concatenate(parts)).cuda(), off, vt.Params(precision=prec, emit=("nbr", "vol", "cen")))
    b.capture()
    b.replay()
    cells = b.result()
    vol = cells.vol.cpu().numpy()
    for i, p in enumerate(parts):
        if len(p):
            np.testing.assert_allclose(vol[off[i]:off[i + 1]], oracle.tessellate(p)["vol"], rtol=TOL[prec])


def test_repeats_bit_for_bit():
    pts = torch.from_numpy(W.mixed(30_011, 33, n_clumps=20)).cuda()
    for prec in ("fp32", "fp64"):
        p = vt.Params(precision=prec, emit=("nbr", "vol", "cen", "m2", "geom"))
        a = vt.tessellate(pts, p)
        for _ in range(3):
            b = vt.tessellate(pts, p)
            for name in ("vol", "cen", "m2", "nbr", "vtx", "face_nbr", "face_vtx"):
                assert torch.equal(getattr(a, name), getattr(b, name)), (prec, name)


@PRECS
@pytest.mark.parametrize("lattice", [False, True])
def test_fused_schedule_in_parts(lattice, prec):
    # three parts of the cloud, four of the lattice; of the lattice every cell fails its certificate, more than the
    # slots that outlive a part. The list schedule builds the same cells at once
    # (but which of the lattice's faces without area it lists is round-off)
    x = torch.from_numpy(W.cubic_lattice(60) if lattice else W.mixed(200_000, 2, n_clumps=100)).cuda()
    emit = ("nbr", "vol", "cen")
    a = vt.tessellate(x, vt.Params(precision=prec, emit=emit))
    b = vt.tessellate(x, vt.Params(precision=prec, emit=emit, fused=True))
    torch.testing.assert_close(b.vol, a.vol, rtol=TOL[prec], atol=0)
    torch.testing.assert_close(b.cen, a.cen, rtol=0, atol=TOL[prec] * float(a.vol.max()) ** (1 / 3))
    if prec == "fp64" and not lattice:
        assert torch.equal(b.nbr_off, a.nbr_off) and torch.equal(b.nbr, a.nbr)
    again = vt.tessellate(x, vt.Params(precision=prec, emit=emit, fused=True, no_sync=True))
    assert torch.equal(again.vol, b.vol) and torch.equal(again.nbr[:int(b.nbr_off[-1])], b.nbr[:int(b.nbr_off[-1])])


def test_retries_and_rechecks_are_counted():
    # a lattice moved by 1e-4 of its spacing has planes within float32 round-off of
    # most cells' vertices, and a shell of 60 generators gives a cell of more than
    # the 48 vertices of a group (beside enough points that groups run)
    rng = np.random.default_rng(2)
    x = W.cubic_lattice(20)
    x = (x + rng.uniform(-1e-4 / 20, 1e-4 / 20, x.shape)).astype(np.float32)
    s = vt.tessellate(torch.from_numpy(x).cuda(), vt.Params(emit=("vol",))).stats
    assert s["fp64_rechecks"] > len(x) // 4 and s["precision_retries"] > len(x) // 100, s
    d = rng.standard_normal((60, 3))
    shell = 0.5 + (0.2 + 1e-3 * rng.random((60, 1))) * d / np.linalg.norm(d, axis=1, keepdims=True)
    far = rng.random((20_000, 3))
    far = far[np.linalg.norm(far - 0.5, axis=1) > 0.42]
    x = torch.from_numpy(np.concatenate([[[0.5, 0.5, 0.5]], shell, far]).astype(np.float32)).cuda()
    for prec in ("fp32", "fp64"):
        s = vt.tessellate(x, vt.Params(precision=prec, emit=("vol",))).stats
        assert s["capacity_retries"] >= 1 and s["unvalidated"] == 0, s
    assert s["fp64_rechecks"] == 0  # (of the FP32 form)


def test_differentiable_moments_free_their_cells():
    # after a step only its gradient is left: the cells are not kept by a cycle
    # between the outputs and their node
    x = torch.from_numpy(W.uniform(20_000, 5)).cuda().requires_grad_(True)
    held = []
    for _ in range(4):
        x.grad = None
        vol, cen, m2 = vt.voronoi_moments(x, vt.Params())
        (m2.sum() + (vol * vol).sum() + cen.sum()).backward()
        del vol, cen, m2
        torch.cuda.synchronize()
        held.append(torch.cuda.memory_allocated())
    assert held[-1] == held[0], held
