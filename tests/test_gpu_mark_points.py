"""Point predicate, block walk: the walk that only marks (faces gathered and tested a lane per face, bins beyond d
left out, nearest rows first) against the walk that keeps every pair, bit for bit on the same level: bins from one
to more rows than a warp has lanes, faces far below and far above d, both searches."""
import numpy as np
import pytest

from tests.test_gpu_face_pass import OFF
from tests.test_gpu_mark_cells import _soup

pytestmark = pytest.mark.gpu


def _masks(dim, v, f, B, d, search, adjacency):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    g = AmrGeom(dim, (4,) * dim)
    g.load(torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda())
    g.bin(B)
    res = g.refine(2, d, 0.0, 0, adjacency, False, predicate=1, search=search, face_pass=OFF)
    torch.cuda.synchronize()
    return [(lv["blocks"].clone(), lv["mask"].clone(), lv["flag"].clone()) for lv in res["levels"]]


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("search", [0, 1])
@pytest.mark.parametrize("B,d", [(1, 0.1), (5, 0.03), (24, 0.15), (40, 0.25)])
@pytest.mark.parametrize("size,snap,n", [(0.002, None, 900), (0.02, 1 / 64, 400), (0.3, None, 40)])
def test_marks_equal_the_full_walk(dim, search, B, d, size, snap, n):
    import torch

    v, f = _soup(dim, size, n, seed=7 * n + B, snap=snap)
    v = (0.3 + 0.4 * v).astype(np.float32) if snap is None else v
    a = _masks(dim, v, f, B, d, search, False)
    b = _masks(dim, v, f, B, d, search, True)
    for x, y in zip(a, b):
        assert all(torch.equal(p, q) for p, q in zip(x, y))
    assert int(a[-1][2].sum()) > 0
