"""Marks with d the cell size: few small faces are tested against every inflated cell (n_face_tests counts these), many
or wide ones against the cells that they meet; the marks are those of the block walk either way."""
import numpy as np
import pytest

from tests.test_gpu_face_pass import OFF, ON

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,cells,widens", [(3, 200, 1.0, False), (3, 200, 4.0, True), (3, 3500, 0.5, True),
                                                (3, 1000, 2.0, True), (2, 2000, 4.0, False), (2, 3500, 4.0, True),
                                                (2, 100, 30.0, True)])
def test_route(dim, n, cells, widens):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    rng = np.random.default_rng(n)
    t = rng.uniform(0.1, 0.9, (n, 1, dim)) + rng.uniform(-0.5, 0.5, (n, dim, dim)) * cells / 128
    dev = torch.from_numpy(t.astype(np.float32)).cuda()
    masks, tests = [], []
    for face_pass in (0, ON, OFF):
        g = AmrGeom(dim, (8,) * dim)
        g.load(dev)
        g.bin(16)
        r = g.refine(3, 0.0, 1.0, 0, False, False, face_pass=face_pass)
        masks.append(torch.cat([lv["mask"] for lv in r["levels"]]))
        tests.append(r["n_face_tests"])
        g.close()
    assert torch.equal(masks[0], masks[1]) and torch.equal(masks[0], masks[2])
    assert tests[2] == 0 and (tests[0] == tests[1] if widens else tests[0] > tests[1])
