"""Links found from the faces at other distances than the cell size, and with the point predicate, against the
pair kernel: every output identical bit for bit (the walk's lists, or the faces' marks on the levels above)."""
import numpy as np
import pytest

from tests.test_gpu_face_links import OFF, ON, _faces

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["sphere", "box_centres", "copies"])
@pytest.mark.parametrize("pred,d_rel", [(0, 0.51), (0, 0.75), (0, 1.5), (0, 2.5), (1, 1.45)])
def test_face_links_equal_pairs(kind, pred, d_rel):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    t, root, levels, bins = _faces(kind)
    if kind == "copies":  # (pairs enough for the path that is tested)
        t = np.tile(t, (8 if d_rel < 1 else 2, 1, 1))
    elif d_rel < 1:
        root = 4 * root
    dev = torch.from_numpy(np.ascontiguousarray(t)).cuda()
    outs = []
    for face_pass, graph in ((ON, False), (ON, True), (OFF, False)):
        g = AmrGeom(3, (root,) * 3)
        g.load(dev)
        g.bin(bins)
        for _ in range(2 if graph else 1):
            r = g.refine(levels, 0.0, d_rel, 19, True, True, predicate=pred, use_graph=graph, face_pass=face_pass)
        assert r["graph_replay"] == graph
        assert r["adj_ids"].numel() >= (12 if d_rel < 1 else 4) << 20
        outs.append({k: r[k].clone() for k in ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_dir", "link_q",
                                               "link_face")})
        g.close()
    for o in outs[1:]:
        assert all(torch.equal(outs[0][k], o[k]) for k in outs[0])
    assert outs[0]["link_q"].numel() > 0
