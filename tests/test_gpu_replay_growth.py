"""A captured level loop replayed on a geometry that needs far more room than the one it was captured on: the replay
reports that its capacities were outgrown without reading past them, the call runs again eagerly, and the outputs are
those of a fresh context."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_dir", "link_q", "link_face")


def _call(g, verts, bins, levels, graph):
    import torch

    before = g.launch_count()
    g.load(torch.from_numpy(verts).cuda())
    g.bin(bins)
    r = g.refine(levels, 0.0, 1.0, 19, True, True, use_graph=graph, face_pass=2)
    out = [lv[k].clone() for lv in r["levels"] for k in ("blocks", "mask", "flag")] + [r[k].clone() for k in KEYS]
    return out, r["graph_replay"], g.launch_count() - before


def _grow(small, large, root, bins, levels):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    g, fresh = AmrGeom(3, (root,) * 3), AmrGeom(3, (root,) * 3)
    _call(g, small, bins, levels, True)
    assert _call(g, small, bins, levels, True)[1]
    want, _, eager = _call(fresh, large, bins, levels, False)
    for replayed in (False, True):
        got, replay, launches = _call(g, large, bins, levels, True)
        assert replay == replayed
        assert replayed or launches >= eager + 10, "the captured loop was not tried"  # its own launches come on top
        for a, b in zip(got, want):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    g.close()
    fresh.close()


def _tiny(rng, n, lo, hi):
    return rng.uniform(lo, hi, (n, 1, 3)) + rng.normal(0, 1e-3, (n, 3, 3))


def test_more_records_than_staged():
    """64 blocks stage 1,280 records; 4,000 faces, at first 3,500 of them outside the domain, leave over 4,000."""
    rng = np.random.default_rng(1)
    inside = _tiny(rng, 500, 0.1, 0.9)
    small = np.concatenate([inside, _tiny(rng, 3500, 1.5, 1.9)]).astype(np.float32)
    large = np.concatenate([inside, _tiny(rng, 3500, 0.3, 0.5)]).astype(np.float32)
    _grow(small, large, 4, 2, 1)


@pytest.mark.parametrize("levels", [2, 4])
def test_more_blocks_than_captured(levels):
    """600 faces in one corner, then all over the domain: every level below the roots has many times its blocks, and
    the faces look their blocks up through the levels above."""
    rng = np.random.default_rng(2)
    small = _tiny(rng, 600, 0.02, 0.1).astype(np.float32)
    large = _tiny(rng, 600, 0.02, 0.98).astype(np.float32)
    _grow(small, large, 8, 2, levels)


def test_more_hits_than_captured():
    """Links found from the faces (over 4 M pairs): a sphere beside a copy of itself outside the domain, then on top of
    it.  The cells stay, every link is hit twice."""
    from synth import geometry as G

    v, f = G.jittered_sphere(6, radius=0.3, centre=(0.5, 0.49, 0.51), sigma=1e-4, seed=9)
    t = v[f]
    small, large = np.concatenate([t, t + np.float32(2.0)]), np.concatenate([t, t])
    _grow(small.astype(np.float32), large.astype(np.float32), 32, 8, 3)
