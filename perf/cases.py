"""The performance cases of the near-wall refinement library.

Each case is one call sequence that a user of the library runs in earnest, through
``AmrGeom``, ``AmrBatch`` and ``q_links``.  The sizes are those of the repository's workloads
(``synth/configs.py``): a 2D polygon, spheres and bumpy closed surfaces of 20 thousand to 1.3
million triangles on 16^3 to 64^3 root blocks, the paper's 2D and 3D setups, and a batch of uneven
geometries.  ``draw`` gives more cases of the same ranges.

A case's ``kind`` is the call sequence:

  step      load -> bin -> refine with adjacency lists and wall links
  grad      ``q_links`` and the backward pass of a loss on q, to the vertex coordinates
  moving    two positions of a wall: step, step with the previous hierarchy kept, re-adaptation maps
  fluid     step, node classification, restriction of the links to the fluid nodes
  faces     cells whose centre lies within a fixed distance of the wall, with or without their face
            lists (``lists``), no links
  paper     the paper's own search: sampled bins, own bin only, mark propagation
  batch     several geometries in one ``AmrBatch``: run, gradient of a loss on q, per-geometry views

A case has one body; the seed turns it (the axes change places) and renumbers its vertices and faces,
so inputs of another seed are other inputs with the same number of cells, faces and links.

``graph``: the call asks for replays of the captured level loop (``use_graph``), as a program does
that repeats the step in a time loop; without it every call runs the level loop anew.
``soup``: the mesh comes as a face-vertex list in no particular order (an STL file) instead of an
indexed mesh in the mesher's order.
"""
import functools
import math

import torch

from paper_2502_16310_gb300 import AmrBatch, AmrGeom, q_links

DEV = "cuda"
LOSS_CENTRE = 0.5  # loss on q: sum (q - 1/2)^2 / 2


def listed():
    return [
        # a 2D profile in a small domain: the smallest call, where launches and waits count
        dict(name="circle_2d", kind="step", dim=2, freq=512, amp=0.0, root=16, levels=3, bins=32, d_abs=0.0, d_rel=1.0,
             graph=True, soup=False, lists=True),
        # a sphere prepared once: one-off call on a medium mesh, no graph
        dict(name="sphere_once", kind="step", dim=3, freq=32, amp=0.0, root=32, levels=4, bins=64, d_abs=0.0,
             d_rel=1.0, graph=False, soup=False, lists=True),
        # a moving wall: two time steps and the maps that carry the solver's data across
        dict(name="sphere_moving", kind="moving", dim=3, freq=32, amp=0.0, root=32, levels=4, bins=64, d_abs=0.0,
             d_rel=1.0, graph=True, soup=False, lists=True),
        # preparing the boundary conditions of a flow around a sphere: links of the fluid nodes
        dict(name="sphere_fluid", kind="fluid", dim=3, freq=32, amp=0.0, root=32, levels=4, bins=64, d_abs=0.0,
             d_rel=1.0, graph=False, soup=False, lists=True),
        # a deforming body in a time loop, 82 thousand triangles, five levels
        dict(name="body_step", kind="step", dim=3, freq=64, amp=0.05, root=32, levels=5, bins=128, d_abs=0.0,
             d_rel=1.0, graph=True, soup=False, lists=True),
        # shape optimisation on the same body: q and its vertex gradient
        dict(name="body_grad", kind="grad", dim=3, freq=64, amp=0.05, root=32, levels=5, bins=128, d_abs=0.0,
             d_rel=1.0, graph=False, soup=False, lists=True),
        # the largest mesh of a production run, as a triangle soup
        dict(name="large_step", kind="step", dim=3, freq=256, amp=0.05, root=64, levels=6, bins=256, d_abs=0.0,
             d_rel=1.0, graph=True, soup=True, lists=True),
        # shape optimisation on the largest mesh
        dict(name="large_grad", kind="grad", dim=3, freq=256, amp=0.05, root=64, levels=6, bins=256, d_abs=0.0,
             d_rel=1.0, graph=False, soup=False, lists=True),
        # the paper's 3D setup: refine every cell whose centre lies within 0.05 of the surface, exact search
        dict(name="paper_3d_exact", kind="faces", dim=3, freq=75, amp=0.05, root=16, levels=3, bins=16, d_abs=0.05,
             d_rel=0.0, graph=True, soup=False, lists=False),
        # the same with the paper's sampled bins, own-bin search and mark propagation
        dict(name="paper_3d_sampled", kind="paper", dim=3, freq=75, amp=0.05, root=16, levels=3, bins=16, d_abs=0.05,
             d_rel=0.0, graph=True, soup=False, lists=False),
        # the paper's 2D profile (12,800 edges on 256^2 cells) with every cell's faces within 0.02: long lists
        dict(name="wide_band_2d", kind="faces", dim=2, freq=12800, amp=0.0, root=64, levels=3, bins=16, d_abs=0.02,
             d_rel=0.0, graph=True, soup=False, lists=True),
        # a set of uneven shapes in one batch (a design study): forward and gradient
        dict(name="batch_mixed", kind="batch", dim=3, freq=48, amp=0.05, root=24, levels=4, bins=64, d_abs=0.0,
             d_rel=1.0, graph=True, soup=False, lists=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "grad", "grad", "moving", "fluid", "faces", "paper", "batch", "step2", "grad2",
                       "faces2"])
    c = dict(kind=kind.rstrip("2"), dim=2 if kind.endswith("2") else 3, amp=rng.choice([0.0, 0.03, 0.05]), d_abs=0.0,
             d_rel=rng.choice([0.75, 1.0, 1.0, 1.0, 1.5]), graph=rng.random() < 0.5, soup=rng.random() < 0.3,
             lists=True)
    if c["dim"] == 2:
        c.update(freq=_log(rng, 97, 20000), root=_log(rng, 10, 96), levels=rng.randint(2, 5), bins=_log(rng, 7, 128))
        if c["kind"] == "faces":
            c.update(d_abs=rng.uniform(0.005, 0.02), d_rel=0.0, levels=rng.randint(2, 3), bins=_log(rng, 4, 24),
                     freq=_log(rng, 500, 12800), root=_log(rng, 24, 64), lists=rng.random() < 0.7)
    elif c["kind"] in ("faces", "paper"):
        c.update(freq=_log(rng, 16, 75), root=_log(rng, 8, 16), levels=rng.randint(2, 3), bins=_log(rng, 6, 20),
                 d_abs=rng.uniform(0.02, 0.05), d_rel=0.0, lists=False)
    else:
        c.update(freq=_log(rng, 6, 180), root=_log(rng, 12, 56), levels=rng.randint(2, 6))
        while 4 * c["root"] << (c["levels"] - 1) > 4096:
            c["levels"] -= 1
        c["bins"] = max(4, min(200, int(c["freq"] * rng.uniform(0.8, 2.2))))
        if c["kind"] == "batch":
            c["freq"], c["levels"] = min(c["freq"], 64), min(c["levels"], 4)
    if c["kind"] in ("grad",):
        c["graph"] = False
    return c


# -- meshes -------------------------------------------------------------------

@functools.lru_cache(maxsize=8)
def _unit_sphere(freq):
    """Geodesic sphere: every icosahedron face split into freq^2 triangles, shared points merged.
    (unit vertices FP64, faces int64), vertices in the order in which the faces name them."""
    p = (1.0 + math.sqrt(5.0)) / 2.0
    c = torch.tensor([[-1, p, 0], [1, p, 0], [-1, -p, 0], [1, -p, 0], [0, -1, p], [0, 1, p], [0, -1, -p], [0, 1, -p],
                      [p, 0, -1], [p, 0, 1], [-p, 0, -1], [-p, 0, 1]], dtype=torch.float64, device=DEV)
    c = c / c.norm(dim=1, keepdim=True)
    f = torch.tensor([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                      [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5],
                      [2, 4, 11], [6, 2, 10], [8, 6, 7], [9, 8, 1]], device=DEV)
    n = freq
    g = torch.arange(n + 1, device=DEV)
    i, j = torch.meshgrid(g, g, indexing="ij")
    keep = (i + j) <= n
    lut = torch.full((n + 1, n + 1), -1, dtype=torch.int64, device=DEV)
    lut[keep] = torch.arange(int(keep.sum()), device=DEV)
    i, j = i[keep], j[keep]
    w = torch.stack([n - i - j, i, j], 1)  # weights of the face's three corners
    up = (g[:-1, None] + g[None, :-1]) < n
    a, b = torch.nonzero(up, as_tuple=True)
    tri_up = torch.stack([lut[a, b], lut[a + 1, b], lut[a, b + 1]], 1)
    a, b = torch.nonzero((g[:-1, None] + g[None, :-1]) < n - 1, as_tuple=True)
    tri_dn = torch.stack([lut[a + 1, b], lut[a + 1, b + 1], lut[a, b + 1]], 1)
    tri = torch.cat([tri_up, tri_dn])
    tri = tri[torch.argsort(tri.amin(1), stable=True)]  # row by row
    # one key per point, the same from every face that has it (a zero weight drops the corner)
    h = torch.tensor([pow(0x9E3779B97F4A7C15, k + 3, 1 << 61) for k in range(12)], dtype=torch.int64, device=DEV)
    key = (w[None] * h[f][:, None, :]).sum(2).reshape(-1)
    pos = (w[None, :, :, None].double() * c[f][:, None]).sum(2).reshape(-1, 3)
    tris = (tri[None] + (torch.arange(20, device=DEV) * w.shape[0])[:, None, None]).reshape(-1, 3)
    uniq, inv = torch.unique(key, return_inverse=True)
    first = torch.full_like(uniq, key.numel()).scatter_reduce_(0, inv, torch.arange(key.numel(), device=DEV), "amin")
    order = torch.argsort(first)
    rank = torch.empty_like(order)
    rank[order] = torch.arange(order.numel(), device=DEV)
    pos = pos[first[order]]
    return pos / pos.norm(dim=1, keepdim=True), rank[inv][tris]


def _mesh(dim, freq, amp, body, seed):
    """(vertices float32, faces int32) on the GPU: a polygon of `freq` edges in 2D, a sphere of
    20 freq^2 triangles in 3D; amp > 0: a smooth bumpy, squashed body instead of a round one.
    `body` shapes it, `seed` turns and renumbers it."""
    gen = torch.Generator().manual_seed(body)
    rnd = lambda *s: torch.rand(*s, generator=gen, dtype=torch.float64)  # noqa: E731
    centre = (0.5 + 0.02 * (rnd(dim) - 0.5)).to(DEV)
    radius = 0.25 * (1.0 + 0.04 * (float(rnd(1)) - 0.5))
    if dim == 2:
        k = torch.arange(freq, device=DEV)
        ang = 2.0 * math.pi * k.double() / freq + float(rnd(1))
        u, f = torch.stack([ang.cos(), ang.sin()], 1), torch.stack([k, (k + 1) % freq], 1)
    else:
        u, f = _unit_sphere(freq)
    r = torch.full((u.shape[0],), radius, dtype=torch.float64, device=DEV)
    scale = torch.ones(dim, dtype=torch.float64, device=DEV)
    if amp > 0:
        m = 24
        k = torch.randn(m, dim, generator=gen, dtype=torch.float64)
        k = k / k.norm(dim=1, keepdim=True) * (1.0 + 9.0 * rnd(m, 1))
        a = torch.randn(m, generator=gen, dtype=torch.float64) * amp / k.norm(dim=1) * 2.0
        a = a * min(1.0, 0.35 / float(a.abs().sum()))
        k, a, ph = k.to(DEV), a.to(DEV), (2.0 * math.pi * rnd(m)).to(DEV)
        r = r * (1.0 + (torch.cos(u @ k.T + ph) * a).sum(1))
        scale = torch.tensor([1.0, 0.8, 0.9][:dim], dtype=torch.float64, device=DEV)
    noise = torch.randn(u.shape, generator=torch.Generator(DEV).manual_seed(body + 1), device=DEV, dtype=torch.float64)
    spacing = radius * (2.0 * math.pi / freq if dim == 2 else 1.1 / freq)
    p = u * r[:, None] * scale + centre + noise * min(1e-4, 0.02 * spacing)
    if dim == 2 and seed % 2:  # mirrored, counter-clockwise again
        p, f = p.flip(1), f.flip(1)
    elif dim == 3:
        p = p.roll(seed % 3, 1)
    turn = torch.Generator().manual_seed(seed)
    k = int(torch.randint(p.shape[0], (1,), generator=turn))
    f = ((f + k) % p.shape[0]).roll(int(torch.randint(f.shape[0], (1,), generator=turn)), 0)
    return p.roll(k, 0).float().contiguous(), f.int().contiguous()


def _soup(v, f, seed):
    """Face-vertex list of an indexed mesh, its faces in random order."""
    order = torch.randperm(f.shape[0], generator=torch.Generator(DEV).manual_seed(seed + 2), device=DEV)
    return v[f[order].long()].contiguous()


def _batch_sizes(case):
    """(freq, root, levels, bins) of the batch's eight geometries, uneven around the case's."""
    out = []
    for i, (s, r, dl) in enumerate([(1.0, 1.0, 0), (0.3, 1.4, -1), (1.8, 0.8, 0), (0.5, 1.0, 1), (0.15, 0.7, 0),
                                    (1.2, 1.3, -1), (0.7, 0.6, 0), (0.4, 0.9, -2)]):
        fr = max(3, int(case["freq"] * s))
        out.append((fr, max(4, int(case["root"] * r)), max(2, case["levels"] + dl), max(4, int(case["bins"] * s))))
    return out


def _inputs(case, seed):
    """The meshes of a case: a list of (vertices, faces or None)."""
    dim, soup = case["dim"], case["soup"]
    if case["kind"] == "batch":
        got = [_mesh(dim, fr, case["amp"], 10 * fr + i, 101 * seed + i)
               for i, (fr, _, _, _) in enumerate(_batch_sizes(case))]
    else:
        got = [_mesh(dim, case["freq"], case["amp"], 10 * case["freq"], seed)]
        if case["kind"] == "moving":  # the next position: a quarter of a finest cell further, not along an axis
            h = 1.0 / (4 * case["root"] << (case["levels"] - 1))
            v, f = got[0]
            step = torch.tensor([1.0, 0.6, 0.3][:dim], device=DEV, dtype=torch.float64)
            step = step.flip(0) if dim == 2 and seed % 2 else step.roll(seed % 3, 0) if dim == 3 else step
            got.append(((v.double() + 0.25 * h * step).float(), f))
    return [(_soup(v, f, 101 * seed + i), None) if soup else (v, f) for i, (v, f) in enumerate(got)]


# -- the calls ------------------------------------------------------------------

def prepare(case, seed):
    s = dict(case=case, meshes=_inputs(case, seed), lattice=9 if case["dim"] == 2 else 19)
    if case["kind"] == "batch":
        s["batch"] = AmrBatch(case["dim"])
        for (v, f), (_, root, levels, bins) in zip(s["meshes"], _batch_sizes(case)):
            s["batch"].add(v, f, root, levels, case["d_abs"], case["d_rel"], bins)
    else:
        s["geom"] = AmrGeom(case["dim"], case["root"])
    return s


def _levels(r):
    return [{"blocks": x["blocks"], "mask": x["mask"], "flag": x["flag"]} for x in r["levels"]]


def _adjacency(r):
    return {k: r[k] for k in ("adj_cell", "adj_off", "adj_ids") if k in r}


def _links(r):
    return {k: r[k] for k in ("link_cell", "link_dir", "link_q", "link_face")}


_HANDLE = [None]  # results are views of the handle's buffers: the last pass's handle outlives its results


def run(s):
    c, lat = s["case"], s["lattice"]
    _HANDLE[0] = s
    if c["kind"] == "batch":
        b = s["batch"]
        b.run(lat, use_graph=c["graph"])
        views = [b.view(i) for i in range(len(s["meshes"]))]
        grad = b.q_backward(_batch_grad(views))
        return {"grad": grad, "geoms": [{**_adjacency(v), **_links(v)} for v in views]}
    g = s["geom"]
    v, f = s["meshes"][0]
    if c["kind"] == "grad":
        x = v.detach().requires_grad_(True)
        q = q_links(g, x, f, c["bins"], c["levels"], c["d_abs"], c["d_rel"], lat)
        (0.5 * (q - LOSS_CENTRE) ** 2).sum().backward()
        return {"q": q.detach(), "grad": x.grad, "links": _links(g.result)}
    g.load(v, f)
    if c["kind"] == "paper":
        g.bin(c["bins"], sampled=True)
        r = g.refine(c["levels"], c["d_abs"], c["d_rel"], want_adjacency=c["lists"], use_graph=c["graph"],
                     predicate=1, search=1, propagate=-1)
        return {"levels": _levels(r), **_adjacency(r)}
    g.bin(c["bins"])
    if c["kind"] == "faces":
        r = g.refine(c["levels"], c["d_abs"], c["d_rel"], want_adjacency=c["lists"], use_graph=c["graph"],
                     predicate=1)
        return {"levels": _levels(r), **_adjacency(r)}
    r = g.refine(c["levels"], c["d_abs"], c["d_rel"], lat, use_graph=c["graph"])
    if c["kind"] == "moving":
        v, f = s["meshes"][1]
        g.load(v, f)
        g.bin(c["bins"])
        r = g.refine(c["levels"], c["d_abs"], c["d_rel"], lat, use_graph=c["graph"], keep_previous=True)
        maps = g.adapt_diff()
        return {"levels": _levels(r), **_adjacency(r), **_links(r), "maps": maps}
    if c["kind"] == "fluid":
        solid, undecided = g.classify()
        r = g.fluid_links()
        return {"solid": solid, "undecided": undecided, **_adjacency(r), **_links(r)}
    return {"levels": _levels(r), **_adjacency(r), **_links(r)}


def _batch_grad(views):
    """dloss/dq in the batch's own link order: geometry i's links start at its link base."""
    out = torch.empty(sum(v["link_q"].numel() for v in views), device=DEV)
    for v in views:
        n, base = v["link_q"].numel(), v["bases"]["link"]
        torch.sub(v["link_q"], LOSS_CENTRE, out=out[base:base + n])
    return out


# -- what a pass cannot do without ----------------------------------------------

def _work_one(dim, freq, amp, root, levels, case, with_links):
    """Bytes of the faces read once and of the outputs written once, counted from the wall's size in
    finest cells, and the operations of the decisions that the outputs hold (an axis test of about
    100 operations per adjacent pair, a plane crossing of about 30 per link)."""
    h = 1.0 / (4 * root << (levels - 1))
    d = case["d_abs"] + case["d_rel"] * h
    nf = freq if dim == 2 else 20 * freq * freq
    area = (2.0 * math.pi * 0.25 if dim == 2 else math.pi * 0.25) * (1.0 if amp == 0 else 0.8)
    wall = area / h ** (dim - 1)                      # the wall in finest cells
    cells = wall * (2.0 * d / h + (0.0 if case["d_abs"] else 2.5))
    reach = (d if case["d_abs"] else 1.6 * (d + 0.5 * h))
    pairs = cells * max(1.0, (nf / area * (3.0 if dim == 3 else 2.0) * reach ** (dim - 1)) + 1.2)
    links = wall * (11.5 if dim == 3 else 5.5) if with_links else 0.0
    if not case["lists"]:  # each near-wall cell is decided by one face
        pairs, cells = cells, cells / 4.0
    out = links * 13 + (pairs * 4 + cells * 8 if case["lists"] else 0) + cells / 20 * (4 * dim + 9)
    return {"bytes": nf * dim * (dim + 1) * 4 + out, "flops": pairs * 100 + links * 30, "links": links, "nf": nf}


def work(case):
    kind, dim = case["kind"], case["dim"]
    parts = []
    sizes = _batch_sizes(case) if kind == "batch" else [(case["freq"], case["root"], case["levels"], case["bins"])]
    for fr, root, levels, _ in sizes:
        parts += [_work_one(dim, fr, case["amp"], root, levels, case, kind not in ("faces", "paper"))]
    if kind == "moving":
        parts = parts * 2
    w = {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    links = sum(p["links"] for p in parts)
    if kind in ("grad", "batch"):  # the links and dloss/dq read once, the gradient written
        w["bytes"] += links * 17 + sum(p["nf"] for p in parts) * dim * 2
        w["flops"] += links * 30
    if kind == "fluid":
        w["bytes"] += links * 13 * 0.5
    return w


# -- the same in 64 bits ----------------------------------------------------------

def _dirs(dim):
    """The lattice lines (one sense each) and, per line, the direction numbers of its two senses."""
    if dim == 2:
        return [((1, 0), 1, 3), ((0, 1), 2, 4), ((1, 1), 5, 7), ((-1, 1), 6, 8)]
    lines = [((1, 0, 0), 1), ((0, 1, 0), 3), ((0, 0, 1), 5), ((1, 1, 0), 7), ((1, -1, 0), 9), ((1, 0, 1), 11),
             ((1, 0, -1), 13), ((0, 1, 1), 15), ((0, 1, -1), 17)]
    return [(d, a, a + 1) for d, a in lines]


def _cell_order(cell, dim, root, levels):
    """Rank key of finest cells in the library's order: root block (x fastest), then the child slots
    from the first level down, then the cell within its block (x fastest)."""
    r = cell[:, 0] * 0
    for a in reversed(range(dim)):
        r = r * root + (cell[:, a] >> (levels + 1))
    for sh in range(levels, 1, -1):
        for a in reversed(range(dim)):
            r = r * 2 + ((cell[:, a] >> sh) & 1)
    for a in reversed(range(dim)):
        r = r * 4 + (cell[:, a] & 3)
    return r


def _exact_links(v, f, dim, root, levels):
    """All wall links in FP64 from the definition: per (cell, direction) the least t in [0, 1] at which
    x + t c h meets a face.  (q, face, cell, direction vector), ordered by cell, then direction."""
    n_ax = 4 * root << (levels - 1)
    h = 1.0 / n_ax
    P = (v[f.long()] if f is not None else v).double()  # [F, dim, dim]
    lo = ((P.amin(1) / h).floor().long() - 2).clamp(0, n_ax - 1)
    hi = ((P.amax(1) / h).floor().long() + 2).clamp(0, n_ax - 1)
    ext = hi - lo + 1
    count = ext.prod(1)
    end = torch.cumsum(count, 0)
    keys, ts, faces = [], [], []
    start, f0, step = 0, 0, 24_000_000  # (face, cell) pairs at a time
    while f0 < P.shape[0]:
        f1 = max(f0 + 1, int(torch.searchsorted(end, start + step, right=True)))
        stop = int(end[f1 - 1])
        fi = torch.repeat_interleave(torch.arange(f0, f1, device=DEV), count[f0:f1])
        k = torch.arange(start, stop, device=DEV) - (end - count)[fi]
        start, f0 = stop, f1
        cell = torch.empty(fi.numel(), dim, dtype=torch.int64, device=DEV)
        for a in range(dim):
            cell[:, a] = lo[fi, a] + k % ext[fi, a]
            k = k // ext[fi, a]
        x = (cell.double() + 0.5) * h
        p0 = P[fi, 0] - x
        if dim == 3:
            n = torch.linalg.cross(P[fi, 1] - P[fi, 0], P[fi, 2] - P[fi, 0])
        else:
            e = P[fi, 1] - P[fi, 0]
            n = torch.stack([e[:, 1], -e[:, 0]], 1)
        num = (p0 * n).sum(1)
        near = num.abs() <= 1.0001 * h * n.abs().sum(1)  # no lattice direction reaches the plane otherwise
        fi, cell, p0, num, n, x = fi[near], cell[near], p0[near], num[near], n[near], x[near]
        p = [p0] + [P[fi, j] - x for j in range(1, dim)]
        for d, plus, minus in _dirs(dim):
            dv = torch.tensor(d, dtype=torch.float64, device=DEV) * h
            den = (n * dv).sum(1)
            t = num / den
            if dim == 3:
                inside = torch.ones_like(t, dtype=torch.bool)
                for a, b in ((1, 2), (2, 0), (0, 1)):
                    inside &= (torch.linalg.cross(p[a], p[b]) * dv).sum(1) / den >= 0
            else:
                sl = (p0[:, 0] * dv[1] - p0[:, 1] * dv[0]) / den
                inside = (sl >= 0) & (sl <= 1)
            for sense, number in ((1.0, plus), (-1.0, minus)):
                ok = inside & (sense * t >= 0) & (sense * t <= 1) & (den != 0)
                keys.append(_cell_order(cell[ok], dim, root, levels) * 32 + number)
                ts.append((sense * t)[ok])
                faces.append(fi[ok])
    key, t, fa = torch.cat(keys), torch.cat(ts), torch.cat(faces)
    o = torch.argsort(t)
    o = o[torch.argsort(key[o], stable=True)]
    key, t, fa = key[o], t[o], fa[o]
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    return t[first], fa[first], key[first]


def _decode(key, dim, root, levels):
    """Cell coordinates and direction vectors of link keys (see _cell_order)."""
    number, r = key % 32, key // 32
    cell = torch.zeros(key.numel(), dim, dtype=torch.int64, device=DEV)
    for a in range(dim):
        cell[:, a] = r % 4
        r = r // 4
    for sh in range(2, levels + 1):
        for a in range(dim):
            cell[:, a] += (r % 2) << sh
            r = r // 2
    for a in range(dim):
        cell[:, a] += (r % root) << (levels + 1)
        r = r // root
    table = torch.zeros(32, dim, dtype=torch.float64, device=DEV)
    for d, plus, minus in _dirs(dim):
        table[plus] = torch.tensor(d, dtype=torch.float64)
        table[minus] = -table[plus]
    return cell, table[number]


def _exact_grad(v, f, q, fa, key, dim, root, levels):
    """Gradient of sum (q - 1/2)^2 / 2 with respect to the vertices, q = num / den of the hit face."""
    h = 1.0 / (4 * root << (levels - 1))
    x = v.double().requires_grad_(True)
    cell, d = _decode(key, dim, root, levels)
    out = torch.zeros_like(x)
    for i in range(0, key.numel(), 20_000_000):
        s = slice(i, i + 20_000_000)
        P = x[f[fa[s]].long()] if f is not None else x[fa[s]]
        p0 = P[:, 0] - (cell[s].double() + 0.5) * h
        if dim == 3:
            n = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
        else:
            e = P[:, 1] - P[:, 0]
            n = torch.stack([e[:, 1], -e[:, 0]], 1)
        t = (p0 * n).sum(1) / (d[s] * h * n).sum(1)
        out += torch.autograd.grad(t, x, q[s] - LOSS_CENTRE)[0]
    return out


def exact(case, seed):
    kind, dim = case["kind"], case["dim"]
    fine = 4 * case["root"] << (case["levels"] - 1)
    if kind in ("faces", "paper", "fluid"):
        return None  # whole numbers, or links picked by the classification
    if dim == 3 and fine > 2100:
        return None  # hundreds of millions of links
    meshes = _inputs(case, seed)
    nothing = {"link_cell": None, "link_dir": None, "link_face": None}
    adj = {"adj_cell": None, "adj_off": None, "adj_ids": None}
    if kind == "batch":
        grads, geoms = [], []
        for (v, f), (_, root, levels, _) in zip(meshes, _batch_sizes(case)):
            q, fa, key = _exact_links(v, f, dim, root, levels)
            grads.append(_exact_grad(v, f, q, fa, key, dim, root, levels))
            geoms.append({**adj, **nothing, "link_q": q})
        return {"grad": torch.cat(grads), "geoms": geoms}
    v, f = meshes[-1]
    q, fa, key = _exact_links(v, f, dim, case["root"], case["levels"])
    if kind == "grad":
        grad = _exact_grad(v, f, q, fa, key, dim, case["root"], case["levels"])
        return {"q": q, "grad": grad, "links": {**nothing, "link_q": q}}
    return {"levels": None, **adj, **nothing, "link_q": q, **({"maps": None} if kind == "moving" else {})}
