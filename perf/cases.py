"""Workloads that stand for what programs do with the Voronoi library.

``listed()`` names them, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes the inputs and what a program keeps between calls (parameters,
workspace, captured batch), ``run`` is one pass through the public entry points,
``work`` the bytes and operations such a pass cannot do without, ``tolerance``
how far two correct implementations may differ and ``exact`` the result in
float64 by plain torch.

Neighbour lists are returned as a table of one row per cell padded with -1, the
form in which graph code takes them: their packed length follows the input, and
in the FP32 form a face at round-off size may be kept by one correct
implementation and dropped by another (about 20 in 100,000 cells), which would
shift everything behind it. Vertex and face order within a cell is not specified, so the
geometry arrays are measured through the call that consumes them all, the
gradient of the cell moments.
"""
import math

import torch

import paper_2412_04514_gb300 as vt
from paper_2412_04514_gb300 import api

# a cell has at most 64 faces (the library refuses more)
TABLE = 64


def listed():
    return [
        # the smallest call: one set of a parameter study, everything at its default
        {"name": "default-1k", "do": "cells", "cloud": "uniform", "n": 1000, "precision": "fp32",
         "emit": "nbr vol cen", "keep": False},
        # the parity configuration: 4,096 uniform points, plain FP64, neighbours, volumes, centroids
        {"name": "uniform-4096-fp64", "do": "cells", "cloud": "uniform", "n": 4096, "precision": "fp64",
         "emit": "nbr vol cen", "keep": True},
        # a small clustered catalogue, all the moments
        {"name": "mixed-10007", "do": "cells", "cloud": "mixed", "n": 10007, "precision": "fp32",
         "emit": "vol cen m2", "keep": True},
        # a simulation snapshot's neighbour graph
        {"name": "mixed-120k-nbr", "do": "cells", "cloud": "mixed", "n": 120011, "precision": "fp32",
         "emit": "nbr vol cen", "keep": True},
        # one training step on the moments of a 1M cloud: tessellation with geometry, adjoint
        {"name": "gradient-1m", "do": "gradient", "cloud": "mixed", "n": 1048576, "precision": "fp32"},
        # the precision configuration's FP64 arm at 1M
        {"name": "mixed-1m-fp64", "do": "cells", "cloud": "mixed", "n": 1048576, "precision": "fp64",
         "emit": "nbr vol cen", "keep": True},
        # the precision configuration's FP32 arm at 8M: densities and centroids
        {"name": "mixed-8m", "do": "cells", "cloud": "mixed", "n": 8388608, "precision": "fp32",
         "emit": "vol cen", "keep": True},
        # many sets of uneven sizes, one captured graph replayed on new coordinates
        {"name": "batch-96", "do": "batch", "sets": 96, "smallest": 1000, "largest": 200000, "precision": "fp32",
         "emit": "vol cen m2"},
        # a periodic simulation box
        {"name": "periodic-262k", "do": "cells", "cloud": "mixed", "n": 262144, "precision": "fp32",
         "emit": "nbr vol cen", "keep": True, "periodic": True},
        # a small periodic box in FP64
        {"name": "periodic-5003-fp64", "do": "cells", "cloud": "uniform", "n": 5003, "precision": "fp64",
         "emit": "nbr vol cen", "keep": True, "periodic": True},
        # the memory-lean schedule
        {"name": "fused-500k", "do": "cells", "cloud": "mixed", "n": 500009, "precision": "fp32",
         "emit": "vol cen", "keep": True, "fused": True},
        # Lloyd relaxation
        {"name": "lloyd-65k", "do": "lloyd", "cloud": "uniform", "n": 65536, "precision": "fp32", "iterations": 2},
    ]


def draw(rng):
    do = rng.choice(["cells", "cells", "cells", "gradient", "batch", "lloyd"])
    precision = rng.choice(["fp32", "fp32", "fp64"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if do == "batch":
        return {"do": do, "sets": size(8, 96), "smallest": size(300, 1500), "largest": size(10000, 100000),
                "precision": precision, "emit": "vol cen m2"}
    cloud = rng.choice(["uniform", "mixed"])
    if do == "lloyd":
        return {"do": do, "cloud": cloud, "n": size(1000, 300000), "precision": precision, "iterations": 2}
    if do == "gradient":
        return {"do": do, "cloud": cloud, "n": size(1000, 700000), "precision": precision}
    c = {"do": do, "cloud": cloud, "n": size(500, 700000), "precision": precision,
         "emit": rng.choice(["nbr vol cen", "vol cen m2"]), "keep": True}
    kind = rng.choice(["plain", "plain", "periodic", "fused"])
    if kind != "plain":
        c[kind] = True
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _uniform(n, g):
    return torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)


def _clumps(n, g, periodic):
    """n points of Gaussian clumps (about 524 each), sigma log-uniform in [1e-3, 1e-2], redrawn or wrapped into the box."""
    m = max(1, -(-n // 524))
    centre = _uniform(m, g)
    sigma = 10.0 ** (-3.0 + torch.rand(m, generator=g, device="cuda", dtype=torch.float64))
    which = torch.randint(0, m, (n,), generator=g, device="cuda")
    x = _uniform(n, g)
    done = torch.zeros(n, 1, dtype=torch.bool, device="cuda")
    for _ in range(1 if periodic else 12):
        y = centre[which] + sigma[which, None] * torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
        if periodic:
            y = y - torch.floor(y)
        y32 = y.float()
        ok = ((y32 >= 0) & (y32 < 1)).all(1, keepdim=True) & ~done
        x = torch.where(ok, y, x)
        done |= ok
    return x


def _cloud(kind, n, g, periodic=False):
    if kind == "uniform":
        x = _uniform(n, g)
    else:
        half = n // 2
        x = torch.cat([_uniform(n - half, g), _clumps(half, g, periodic)])
        x = x[torch.randperm(n, generator=g, device="cuda")]
    x = x.float()
    return torch.where(x >= 1.0, torch.full_like(x, 0.5), x).contiguous()


def _generator(seed):
    return torch.Generator("cuda").manual_seed(int(seed))


def _params(case):
    emit = tuple(case.get("emit", "vol cen m2").split())
    return vt.Params(precision=case["precision"], emit=emit, periodic=bool(case.get("periodic", False)),
                     fused=bool(case.get("fused", False)))


def _sizes(case):
    """Sizes of a batch's sets: the same log-uniform ladder for every seed (a captured graph is kept)."""
    s, a, b = case["sets"], math.log(case["smallest"]), math.log(case["largest"])
    return [int(math.exp(a + (b - a) * ((i * 0.6180339887498949) % 1.0))) for i in range(s)]


def _sets(case, seed):
    g = _generator(seed)
    sizes = _sizes(case)
    pts = torch.cat([_cloud("mixed" if i % 2 else "uniform", n, g) for i, n in enumerate(sizes)])
    off = [0]
    for n in sizes:
        off.append(off[-1] + n)
    return pts, off


def _upstream(n, seed):
    """Gradients of a loss with respect to volumes, centroids and second moments, of comparable effect."""
    g = torch.Generator("cuda").manual_seed(int(seed) + 1000003)
    r = torch.randn(n, 5, generator=g, device="cuda", dtype=torch.float64)
    return r[:, 0].contiguous(), (n ** (-2.0 / 3.0) * r[:, 1:4]).contiguous(), (n ** (2.0 / 3.0) * r[:, 4]).contiguous()


def prepare(case, seed):
    p = _params(case)
    if case["do"] == "batch":
        pts, off = _sets(case, seed)
        b = vt.Batch(pts, off, p)
        b.capture()
        torch.cuda.current_stream().synchronize()
        return {"do": "batch", "points": pts, "batch": b}
    n = case["n"]
    pts = _cloud(case["cloud"], n, _generator(seed), bool(case.get("periodic", False)))
    s = {"do": case["do"], "points": pts, "params": p}
    if case["do"] == "gradient":
        s["up"] = _upstream(n, seed)
    elif case["do"] == "lloyd":
        s["iterations"] = case["iterations"]
    else:
        s["ws"] = api.Workspace(p, n) if case["keep"] else None
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _neighbour_table(cells):
    """The neighbour lists as one row of TABLE ids per cell, padded with -1."""
    off = cells.nbr_off
    at = off[:-1, None] + torch.arange(TABLE, device=off.device)
    ids = torch.take(cells.nbr, at.clamp_(max=cells.nbr.numel() - 1))
    return ids.masked_fill_(at >= off[1:, None], -1) if cells.nbr.numel() else ids


def run(state):
    if state["do"] == "batch":
        b = state["batch"]
        b.points.copy_(state["points"])
        b.replay()
        c = b.result()
        return {"vol": c.vol, "cen": c.cen, "m2": c.m2}
    if state["do"] == "gradient":
        q = state["points"].detach().requires_grad_(True)
        out = vt.voronoi_moments(q, state["params"])
        (grad,) = torch.autograd.grad(out, q, state["up"])
        return {"vol": out[0].detach(), "cen": out[1].detach(), "m2": out[2].detach(), "grad": grad}
    if state["do"] == "lloyd":
        return {"points": vt.lloyd(state["points"], state["iterations"], state["params"])}
    c = vt.tessellate(state["points"], state["params"], workspace=state["ws"])
    out = {"vol": c.vol, "cen": c.cen}
    if c.m2 is not None:
        out["m2"] = c.m2
    if c.nbr is not None:
        out["nbr"] = _neighbour_table(c)
    return out


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------
def work(case):
    """Points read and outputs written once. Operations of a cell known in advance: 16 faces and 27 vertices on average,
    8 for the distance of each of about 60 generators within twice its radius, 60 to solve each vertex, 45 for each of
    the 81 corner terms of the moments."""
    n = sum(_sizes(case)) if case["do"] == "batch" else case["n"]
    cell = 60 * 8 + 27 * 60 + 81 * 45
    if case["do"] == "lloyd":
        return {"bytes": 24 * n * case["iterations"], "flops": cell * n * case["iterations"]}
    if case["do"] == "gradient":
        # (the adjoint: a 7-point rule of about 50 operations on each of the 81 face triangles)
        return {"bytes": n * (12 + 8 * 5 + 8 * 5 + 12), "flops": n * (cell + 81 * 350)}
    emit = case["emit"].split()
    per = 12 + (8 if "vol" in emit else 0) + (24 if "cen" in emit else 0) + (8 if "m2" in emit else 0)
    per += (8 + 4 * 16) if "nbr" in emit else 0
    return {"bytes": per * n, "flops": cell * n}


def tolerance(case):
    """About four times what the two schedules of the library, and its two forms, differ by on these inputs. FP32 form:
    coordinates relative to the generator carry 6e-8 of the cell's size (volumes seen 6e-8 in the 2-norm, 5e-6 in the
    worst cell; gradients 5e-7 and 2e-4). FP64 form: 1e-16 and 7e-15; its gradients, and all points, round to float32."""
    if case["do"] == "lloyd":
        return {"rel": 5e-8, "max": 1e-6}
    if case["do"] == "gradient":
        return {"rel": 1e-7, "max": 1e-6} if case["precision"] == "fp64" else {"rel": 2e-6, "max": 1e-3}
    if case["precision"] == "fp64":
        return {"rel": 1e-14, "max": 2e-13, "differ": 1e-5}
    return {"rel": 4e-7, "max": 2e-5, "differ": 1e-4}


# ---------------------------------------------------------------------------
# the same results in float64 by enumeration, in plain torch
# ---------------------------------------------------------------------------
def _triples(m, dev):
    t = torch.combinations(torch.arange(m, device=dev), 3)
    return t[:, 0], t[:, 1], t[:, 2]


def _solve(A, a, B, b, C, c):
    bc, ca, ab = torch.linalg.cross(B, C), torch.linalg.cross(C, A), torch.linalg.cross(A, B)
    det = (A * bc).sum(-1)
    return (a[..., None] * bc + b[..., None] * ca + c[..., None] * ab) / det[..., None], det


def _corners(nrm, off):
    """Vertices of the intersection of the half-spaces nrm.x <= off of each row: (row, three plane indices) of each."""
    rows, m = off.shape
    i, j, k = _triples(m, off.device)
    size = nrm.norm(dim=-1)
    got = []
    step = max(1, int(1.5e8 // (i.numel() * m)))
    for r in range(0, rows, step):
        N, o, sz = nrm[r:r + step], off[r:r + step], size[r:r + step]
        v, det = _solve(N[:, i], o[:, i], N[:, j], o[:, j], N[:, k], o[:, k])
        good = det.abs() > 1e-10 * sz[:, i] * sz[:, j] * sz[:, k]
        v = torch.where(good[..., None], v, torch.full_like(v, 1e30))
        worst = torch.full_like(det, -1.0)
        for f in range(m):
            s = (v * N[:, f, None, :]).sum(-1) - o[:, f, None]
            s = torch.where((i == f) | (j == f) | (k == f), torch.full_like(s, -1.0), s)
            worst = torch.maximum(worst, s)
        row, t = torch.nonzero(good & (worst <= 0), as_tuple=True)
        got.append(torch.stack([row + r, i[t], j[t], k[t]], 1))
    return torch.cat(got)


def _topology(x, others, wall_off, wall_nrm, own):
    """For every generator the plane ids (an index into `others`, or -1..-6 for a wall) of each vertex of its cell.
    Grows each row's plane set until no generator lies inside the sphere of a vertex."""
    n, dev = len(x), x.device
    cells, planes = [], []
    step = max(8, int(2.5e8 // (len(others) * 40)))
    for r in range(0, n, step):
        xi = x[r:r + step]
        d2 = torch.stack([((others - q) ** 2).sum(1) for q in xi]) if len(others) > 50000 else \
            ((others[None] - xi[:, None]) ** 2).sum(-1)
        d2[torch.arange(len(xi), device=dev), own[r:r + step]] = math.inf
        ids = torch.topk(d2, min(22, len(others) - 1), largest=False).indices
        walls = torch.arange(-1, -7, -1, device=dev).expand(len(xi), 6)
        ids = torch.cat([ids, walls], 1)
        for _ in range(400):
            pad = ids == -100
            wall = (ids < 0) & ~pad
            w = (-1 - ids).clamp(0, 5)
            nrm = torch.where(wall[..., None], wall_nrm[w], others[ids.clamp(min=0)] - xi[:, None])
            off = torch.where(wall, wall_off[r:r + step].gather(1, w), 0.5 * (nrm ** 2).sum(-1))
            nrm = torch.where(pad[..., None], torch.zeros_like(nrm), nrm)
            off = torch.where(pad, torch.ones_like(off), off)
            c = _corners(nrm, off)
            row, t = c[:, 0], c[:, 1:]
            P = [nrm[row, t[:, e]] for e in range(3)]
            o = [off[row, t[:, e]] for e in range(3)]
            v, _ = _solve(P[0], o[0], P[1], o[1], P[2], o[2])
            cut = torch.zeros_like(d2, dtype=torch.bool)
            rad = v.norm(dim=1)
            sub = max(1, int(1e8 // len(others)))
            for q in range(0, len(v), sub):
                dist = torch.cdist((v[q:q + sub] + xi[row[q:q + sub]]), others, compute_mode="donot_use_mm_for_euclid_dist")
                a, b = torch.nonzero(dist < rad[q:q + sub, None] * (1 - 1e-10), as_tuple=True)
                cut[row[q:q + sub][a], b] = True
            face = torch.zeros(ids.shape, dtype=torch.bool, device=dev)
            face[row[:, None].expand(-1, 3).reshape(-1), t.reshape(-1)] = True
            have = torch.where(ids >= 0, ids, torch.zeros_like(ids))
            known = torch.zeros_like(cut)
            known.scatter_(1, have, ids >= 0)
            cut &= ~known
            if not cut.any():
                break
            near = torch.topk(torch.where(cut, d2, torch.full_like(d2, math.inf)), 10, largest=False)
            more = torch.where(near.values < math.inf, near.indices, torch.full_like(near.indices, -100))
            ids = torch.cat([torch.where(face, ids, torch.full_like(ids, -100)), more], 1)
            order = torch.argsort((ids == -100).int(), dim=1, stable=True)
            ids = ids.gather(1, order)[:, :max(4, int((ids != -100).sum(1).max()))]
        else:
            raise RuntimeError("no end")
        cells.append(row + r)
        planes.append(ids[row[:, None], t])
    return torch.cat(cells), torch.cat(planes)


def _moments64(x, periodic):
    """(volumes, centroids, second moments) of the Voronoi cells of float64 points x in the unit box, differentiable."""
    n, dev = len(x), x.device
    shift = torch.zeros(1, 3, dtype=torch.float64, device=dev)
    if periodic:
        shift = torch.cartesian_prod(*[torch.tensor([0.0, -1.0, 1.0], dtype=torch.float64, device=dev)] * 3)
    images = (x[None] + shift[:, None]).reshape(-1, 3)
    wall_nrm = torch.zeros(6, 3, dtype=torch.float64, device=dev)
    for a in range(3):
        wall_nrm[2 * a, a], wall_nrm[2 * a + 1, a] = -1.0, 1.0
    if periodic:
        wall_off = torch.full((n, 6), 0.5, dtype=torch.float64, device=dev)
    else:
        wall_off = torch.stack([x[:, 0], 1 - x[:, 0], x[:, 1], 1 - x[:, 1], x[:, 2], 1 - x[:, 2]], 1)
    own = torch.arange(n, device=dev)
    with torch.no_grad():
        cell, ids = _topology(x.detach(), images.detach(), wall_off.detach(), wall_nrm, own)

    def planes(c, k):
        wall, w = k < 0, (-1 - k).clamp(0, 5)
        nrm = torch.where(wall[:, None], wall_nrm[w], images[k.clamp(min=0)] - x[c])
        return nrm, torch.where(wall, wall_off[c, w], 0.5 * (nrm ** 2).sum(1))

    P = [planes(cell, ids[:, e]) for e in range(3)]
    v, det = _solve(P[0][0], P[0][1], P[1][0], P[1][1], P[2][0], P[2][1])
    # edges: two vertices of a cell that share two planes
    big = len(images) + 8
    key, end, third = [], [], []
    for a, b, c in ((0, 1, 2), (0, 2, 1), (1, 2, 0)):
        lo, hi = torch.minimum(ids[:, a], ids[:, b]) + 7, torch.maximum(ids[:, a], ids[:, b]) + 7
        key.append((cell * big + lo) * big + hi)
        end.append(torch.arange(len(cell), device=dev))
        third.append(ids[:, c])
    key, end, third = torch.cat(key), torch.cat(end), torch.cat(third)
    order = torch.argsort(key)
    if not bool((key[order][0::2] == key[order][1::2]).all()):
        raise RuntimeError("degenerate input")
    e1, e2 = order[0::2], order[1::2]
    v1, v2, c = v[end[e1]], v[end[e2]], cell[end[e1]]
    ka, kb = key[e1] // big % big - 7, key[e1] % big - 7
    na, oa = planes(c, ka)
    nb, ob = planes(c, kb)
    nc, _ = planes(c, third[e1])
    sign = torch.sign((torch.linalg.cross(na, nb) * nc).sum(1)).detach()
    vol = x.new_zeros(n)
    first, second = x.new_zeros(n, 3), x.new_zeros(n)
    for nrm, off, sg in ((nb, ob, sign), (na, oa, -sign)):
        q = nrm * (off / (nrm ** 2).sum(1))[:, None]
        dv = sg * (q * torch.linalg.cross(v1, v2)).sum(1) / 6.0
        s = q + v1 + v2
        vol = vol.index_add(0, c, dv)
        first = first.index_add(0, c, dv[:, None] * s / 4.0)
        second = second.index_add(0, c, dv * ((q ** 2).sum(1) + (v1 ** 2).sum(1) + (v2 ** 2).sum(1) + (s ** 2).sum(1)) / 20.0)
    return vol, x + first / vol[:, None], second


def exact(case, seed):
    if case["do"] == "batch":
        if sum(_sizes(case)) > 16000:
            return None
        pts, off = _sets(case, seed)
        parts = [_moments64(pts[a:b].double(), False) for a, b in zip(off[:-1], off[1:])]
        return {"vol": torch.cat([p[0] for p in parts]), "cen": torch.cat([p[1] for p in parts]),
                "m2": torch.cat([p[2] for p in parts])}
    periodic = bool(case.get("periodic", False))
    n = case["n"]
    if n > (5100 if periodic else 10500):
        return None
    x = _cloud(case["cloud"], n, _generator(seed), periodic).double()
    if case["do"] == "lloyd":
        for _ in range(case["iterations"]):
            x = _moments64(x, periodic)[1].float().double()
        return {"points": x}
    if case["do"] == "gradient":
        x.requires_grad_(True)
        out = _moments64(x, periodic)
        (g,) = torch.autograd.grad(out, x, _upstream(n, seed))
        return {"vol": out[0].detach(), "cen": out[1].detach(), "m2": out[2].detach(), "grad": g}
    vol, cen, m2 = _moments64(x, periodic)
    out = {"vol": vol, "cen": cen}
    if "m2" in case["emit"].split():
        out["m2"] = m2
    if "nbr" in case["emit"].split():
        out["nbr"] = None
    return out
