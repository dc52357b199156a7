"""What the faces leave against the walk and the pair kernel, bit for bit, in corners of the sizes: blocks with more
records than a warp sorts at once, a level whose hits outgrow the first guess, and geometries of a batch with origins
and unequal roots whose links are found from the faces."""
import numpy as np
import pytest

from tests.test_gpu_face_pass import OFF, ON

pytestmark = pytest.mark.gpu

KEYS = ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_dir", "link_q", "link_face")


def _both(tris, root, levels, bins):
    """Outputs with and without the face pass: [(tensors, timings)]."""
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    out = []
    for face_pass in (ON, OFF):
        g = AmrGeom(3, (root,) * 3)
        g.load(torch.from_numpy(np.ascontiguousarray(tris, np.float32)).cuda())
        g.bin(bins)
        g.timing(True)
        r = g.refine(levels, 0.0, 1.0, 19, True, True, face_pass=face_pass)
        torch.cuda.synchronize()
        out.append(([lv["mask"].clone() for lv in r["levels"]] + [r[k].clone() for k in KEYS], g.timings()))
        g.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    return out


@pytest.mark.parametrize("n", [64, 65, 1024, 1025, 1500])
def test_long_records(n):
    rng = np.random.default_rng(n)
    t = rng.uniform(0.42, 0.46, (n, 1, 3)) + rng.uniform(-0.003, 0.003, (n, 3, 3))
    (got, times), _ = _both(t, 4, 2, 5)
    assert "place_records" in times
    counts = np.diff(got[3].cpu().numpy().astype(np.int64))
    assert counts.max() > 0.9 * n


def test_more_hits_than_guessed():
    """Triangles 24 cells wide have about 1.9 hits per pair; room is made for 1.25 at first."""
    rng = np.random.default_rng(6)
    w = np.array([[-0.5, -0.5, 0.5], [0.5, 0.5, -0.5], [0.5, -0.5, 0.5]]) * 24 / 512
    (got, times), _ = _both(rng.uniform(0.1, 0.9, (2000, 1, 3)) + w, 32, 3, 32)
    pairs, links = got[5].numel(), got[8].numel()
    assert pairs >= 4 << 20 and links > 1.25 * pairs + 1024
    assert times["links"][1] == 2  # twice: the second time with room for all


def test_batch_links_from_faces():
    import torch

    from paper_2502_16310_gb300 import AmrBatch
    from synth import geometry as G

    views, cands = [], []
    for face_pass in (ON, OFF):
        b = AmrBatch(3)
        for i, (root, origin, h0, levels) in enumerate([((32, 28, 30), (-3.0, 0.7, 11.0), 1.0 / 128, 3),
                                                        ((20, 24, 36), (0.1, -40.0, 0.0), 0.05, 3),
                                                        ((6, 5, 7), (1.0, 2.0, 3.0), 0.25, 2)]):
            v, f = G.jittered_sphere(6 if i < 2 else 3, radius=0.3, centre=(0.0, 0.0, 0.0), sigma=1e-4, seed=30 + i)
            size = 4 * h0 * np.array(root)
            v = (np.array(origin) + size / 2 + v.astype(np.float64) * size).astype(np.float32)
            b.add(torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda(), root, levels, 0.0, 1.0, 24, origin, h0)
        r = b.run(19, face_pass=face_pass)
        assert int(r.n_adj_pairs) >= 8 << 20
        cands.append(int(r.n_link_candidates))
        views.append([b.view(i) for i in range(3)])
        b.close()
    assert cands[0] != cands[1]
    for x, y in zip(*views):
        assert all(torch.equal(x[k].view(torch.uint8), y[k].view(torch.uint8)) for k in KEYS) and x["link_q"].numel() > 0
