"""A domain far from the coordinates' origin (2^21 finest cells, coordinates a quarter of a cell apart): the faces'
cell ranges are widened by several cells there, and faces that near the origin would just fit the face-driven kernels
are left to the walk and the pair kernel.  Every choice of the face pass gives the same outputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KEYS = ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_dir", "link_q", "link_face")


@pytest.mark.parametrize("cells,n", [(3.0, 60000), (25.0, 8000)])
def test_face_pass_far_from_the_origin(cells, n):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    h = 1.0 / 256
    origin = np.array([8192.0, -8192.0, 4096.0])
    rng = np.random.default_rng(4)
    c = rng.uniform(0.1, 0.9, (n, 1, 3))
    t = rng.uniform(-0.5, 0.5, (n, 3, 3))
    t[:50] = [[-0.5, -0.5, 0.5], [0.5, 0.5, -0.5], [0.5, -0.5, 0.5]]  # as wide as they may be on every axis
    t = c + t * cells * h
    dev = torch.from_numpy((origin + t).astype(np.float32)).cuda()
    outs = []
    for face_pass in (0, 1, 2):  # as the library chooses, off, on
        g = AmrGeom(3, (16,) * 3, origin=tuple(origin), h0=1.0 / 64)
        g.load(dev)
        g.bin(32)
        r = g.refine(3, 0.0, 1.0, 19, True, True, face_pass=face_pass)
        assert r["adj_ids"].numel() >= 4 << 20
        outs.append([lv["mask"].clone() for lv in r["levels"]] + [r[k].clone() for k in KEYS])
        g.close()
    for o in outs[1:]:
        for a, b in zip(outs[0], o):
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
