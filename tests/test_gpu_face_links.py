"""Links found from the faces (levels with millions of (cell, face) pairs) against the pair kernel: every output
identical bit for bit.  A sphere; boxes on cell planes, on planes through the cell centres (crossings exactly on
nodes, decided in FP64) and a hair off them (lattice lines nearly parallel to the faces); and many copies of an
odd soup across the domain's sides (several faces compete for a link, the least face id wins a tie)."""
import numpy as np
import pytest

from synth import geometry as G

pytestmark = pytest.mark.gpu

ON, OFF = 2, 1


def _box(lo, hi, m):
    """Surface of the box [lo, hi]^3, every side m x m squares of two triangles."""
    g = np.linspace(0.0, 1.0, m + 1)
    a, b = np.meshgrid(g[:-1], g[:-1], indexing="ij")
    s = g[1]
    quad = np.stack([np.stack([a, b], -1), np.stack([a + s, b], -1), np.stack([a + s, b + s], -1),
                     np.stack([a, b + s], -1)], -2).reshape(-1, 4, 2)
    out = []
    for axis in range(3):
        for side in (0.0, 1.0):
            q = np.insert(quad, axis, side, axis=2)
            q = q[:, ::-1] if (axis == 1) == (side == 1.0) else q  # outward
            out += [q[:, [0, 1, 2]], q[:, [0, 2, 3]]]
    return (lo + (hi - lo) * np.concatenate(out)).astype(np.float32)


def _faces(kind):
    h = 1.0 / 512
    if kind == "sphere":
        v, f = G.jittered_sphere(6, radius=0.3, centre=(0.5, 0.49, 0.51), sigma=1e-4, seed=9)
        return v[f], 32, 3, 64
    if kind == "box_planes":
        return _box(0.25, 0.75, 64), 32, 3, 32
    if kind == "box_centres":
        return _box(0.25 + h / 2, 0.75 + h / 2, 64), 32, 3, 32
    if kind == "box_tilted":
        t = _box(0.25, 0.75, 64).astype(np.float64)
        t[..., 0] += 3e-6 * t[..., 1]
        t[..., 2] -= 2e-6 * t[..., 0]
        return t.astype(np.float32), 32, 3, 32
    rng = np.random.default_rng(5)
    sizes = np.exp(rng.uniform(np.log(0.002), np.log(0.05), (600, 1, 1)))
    t = rng.uniform(-0.05, 1.05, (600, 1, 3)) + sizes * rng.uniform(-1, 1, (600, 3, 3))
    t = np.repeat(t, 60, axis=0)
    return t[rng.permutation(t.shape[0])].astype(np.float32), 16, 3, 24


@pytest.mark.parametrize("kind", ["sphere", "box_planes", "box_centres", "box_tilted", "copies"])
def test_face_links_equal_pairs(kind):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    t, root, levels, bins = _faces(kind)
    dev = torch.from_numpy(np.ascontiguousarray(t)).cuda()
    outs = []
    for face_pass, graph in ((ON, False), (ON, True), (OFF, False)):
        g = AmrGeom(3, (root,) * 3)
        g.load(dev)
        g.bin(bins)
        for _ in range(2 if graph else 1):
            r = g.refine(levels, 0.0, 1.0, 19, True, True, use_graph=graph, face_pass=face_pass)
        assert r["graph_replay"] == graph
        assert r["adj_ids"].numel() >= 4 << 20
        outs.append({k: r[k].clone() for k in ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_dir", "link_q",
                                               "link_face")})
        g.close()
    for o in outs[:2]:
        for k, x in o.items():
            assert torch.equal(x.view(torch.uint8), outs[2][k].view(torch.uint8)), k
    assert outs[0]["link_q"].numel() > 0
