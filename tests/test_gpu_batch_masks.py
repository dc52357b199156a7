"""A batch that wants masks only (no adjacency was ever made in it) gives the masks of one that wants lists."""
import pytest

from tests.test_gpu_face_pass import OFF
from tests.test_gpu_mark_cells import _soup

pytestmark = pytest.mark.gpu


def test_batch_marks_equal_the_full_walk():
    import torch

    from paper_2502_16310_gb300 import AmrBatch

    outs = []
    for adjacency in (False, True):
        b = AmrBatch(3)
        for i, (d, root, B) in enumerate([(0.05, 4, 9), (0.2, 3, 30), (0.02, 5, 4)]):
            v, f = _soup(3, 0.03, 150 + 37 * i, seed=90 + i)
            b.add(torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda(), root, 2 + (i == 1), d, 0.0, B)
        b.run(0, want_adjacency=adjacency, predicate=1, face_pass=OFF)
        outs.append([b.view(i) for i in range(3)])
    for x, y in zip(*outs):
        for p, q in zip(x["levels"], y["levels"]):
            assert all(torch.equal(p[k], q[k]) for k in ("blocks", "mask", "flag"))
