"""Last level, d the cell size: whether the faces leave its records (a "place_records" launch) or the parents' walk
finds them, as the library chooses and as it is told; the lists are the same."""
import numpy as np
import pytest

from tests.test_gpu_face_pass import OFF, ON

pytestmark = pytest.mark.gpu


def _soup(n, cells, wide, width):
    """n faces of about `cells` cells, then `wide` of exactly `width`, on 256 finest cells per axis."""
    rng = np.random.default_rng(n + wide)
    t = rng.uniform(0.1, 0.9, (n, 1, 3)) + rng.uniform(-0.5, 0.5, (n, 3, 3)) * cells / 256
    w = np.array([[-0.5, -0.5, 0.5], [0.5, 0.5, -0.5], [0.5, -0.5, 0.5]]) * width / 256
    return np.concatenate([t, rng.uniform(0.2, 0.8, (wide, 1, 3)) + w]).astype(np.float32)


@pytest.mark.parametrize("n,cells,wide,width,by_faces", [(40, 2, 0, 0, True), (300, 25, 0, 0, False),
                                                         (5000, 2, 10, 12, True), (5000, 2, 10, 20, False),
                                                         (60000, 1, 2, 20, False), (170000, 1, 2, 20, True)])
def test_route(n, cells, wide, width, by_faces):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    dev = torch.from_numpy(_soup(n, cells, wide, width)).cuda()
    outs = []
    for face_pass, want in ((0, by_faces), (OFF, False), (ON, True)):
        g = AmrGeom(3, (16,) * 3)
        g.load(dev)
        g.bin(32)
        g.timing(True)
        r = g.refine(3, 0.0, 1.0, 19, True, True, face_pass=face_pass)
        torch.cuda.synchronize()
        assert ("place_records" in g.timings()) == want
        outs.append([r[k].clone() for k in ("adj_cell", "adj_off", "adj_ids", "link_face", "link_q")])
        g.close()
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
