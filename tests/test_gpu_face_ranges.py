"""Face-by-face levels of a batch take the faces of the geometries that reach the level: the deepest geometry
first, in the middle and last, alone on its level or with others, against the block walk."""
import pytest

from tests.test_gpu_face_pass import OFF, ON
from tests.test_gpu_mark_cells import _soup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("levels", [(4, 2, 3), (2, 4, 3), (2, 3, 4), (1, 3, 1), (3, 1, 3)])
def test_depths_equal_block_walk(dim, levels):
    import torch

    from paper_2502_16310_gb300 import AmrBatch

    outs = []
    for face_pass in (ON, OFF):
        b = AmrBatch(dim)
        for i, n in enumerate(levels):
            v, f = _soup(dim, 0.03, 90 + 61 * i, seed=20 + i)
            b.add(torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda(), 3 + i, n, 0.0, 1.0, 5)
        b.run(9 if dim == 2 else 19, face_pass=face_pass)
        outs.append([b.view(i) for i in range(len(levels))])
    for x, y in zip(*outs):
        for p, q in zip(x["levels"], y["levels"]):
            assert all(torch.equal(p[k], q[k]) for k in ("blocks", "mask", "flag"))
        assert all(torch.equal(x[k], y[k]) for k in ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_q"))
        assert x["adj_cell"].numel() > 0
