"""Which link kernel a large level takes: even meshes go by their faces, a mesh with a few wide faces among small ones
by its pairs (n_link_candidates counts hits on the first way, queued candidates on the second, so the two differ); the
links are the same."""
import numpy as np
import pytest

from tests.test_gpu_face_pass import OFF, ON
from tests.test_gpu_records_route import _soup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cells,wide,width,by_faces", [(100000, 2, 0, 0, True), (150000, 2, 20, 10, True),
                                                         (100000, 2, 20, 20, False), (14000, 12, 1500, 12, True)])
def test_route(n, cells, wide, width, by_faces):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    dev = torch.from_numpy(_soup(n, cells, wide, width)).cuda()
    cands, outs = [], []
    for face_pass in (0, OFF, ON):
        g = AmrGeom(3, (16,) * 3)
        g.load(dev)
        g.bin(32)
        r = g.refine(3, 0.0, 1.0, 19, True, True, face_pass=face_pass)
        assert r["adj_ids"].numel() >= 4 << 20
        cands.append(r["n_link_candidates"])
        outs.append([r[k].clone() for k in ("adj_ids", "link_cell", "link_dir", "link_face", "link_q")])
        g.close()
    assert cands[1] != cands[2] and cands[0] == cands[2 if by_faces else 1]
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
