"""Face-by-face marking where d is the cell size (the cells that a face meets, widened by one cell) against
the block walk: every output identical.  Soups that sit where the widening can go wrong: across and outside
the domain's sides, on cell and block planes (exact contact, not certified in FP32), from far below a cell to
hundreds of blocks wide, on power-of-two and other grids; and a batch that mixes it with other distances."""
import numpy as np
import pytest

from synth import Workload
from tests import gpu_util as U
from tests.test_gpu_face_pass import OFF, ON, _same

pytestmark = pytest.mark.gpu


def _soup(dim, size, n, seed, snap=None):
    """n random faces with corners within `size` of a centre in [-0.1, 1.1]^dim, corners snapped to a grid."""
    rng = np.random.default_rng(seed)
    v = rng.uniform(-0.1, 1.1, (n, 1, dim)) + rng.uniform(-size, size, (n, dim, dim))
    if snap:
        v = np.round(v / snap) * snap
    v = v.astype(np.float32).reshape(-1, dim)
    return v, np.arange(v.shape[0], dtype=np.int32).reshape(-1, dim)


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("root", [4, 5])
@pytest.mark.parametrize("size,snap", [(0.001, None), (0.02, None), (0.14, None), (0.3, None), (0.05, 1 / 64), (0.05, 1 / 40)])
def test_cells_equal_block_walk(dim, root, size, snap):
    n = 40 if size > 0.2 else 300
    v, f = _soup(dim, size, n, seed=int(1000 * size) + root, snap=snap)
    w = Workload("soup", dim, v, f, root=root, n_levels=3, bins=6, lattice=9 if dim == 2 else 19)
    on = U.run_gpu(w, face_pass=ON)
    off = U.run_gpu(w, face_pass=OFF)
    _same(on, off)
    assert on["n_face_setups"] > 0
    assert sum(int(lv["flag"].sum()) for lv in on["levels"][:-1]) > 0


def test_batch_mixes_distances():
    import torch

    from paper_2502_16310_gb300 import AmrBatch

    outs = []
    for face_pass in (ON, OFF):
        b = AmrBatch(3)
        for i, (d_rel, root) in enumerate([(1.0, 4), (0.75, 5), (1.0, 6), (2.0, 3)]):
            v, f = _soup(3, 0.03, 200 + 37 * i, seed=50 + i)
            b.add(torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda(), root, 3, 0.0, d_rel, 6)
        b.run(19, face_pass=face_pass)
        outs.append([b.view(i) for i in range(4)])
        torch.cuda.synchronize()
    for x, y in zip(*outs):
        for p, q in zip(x["levels"], y["levels"]):
            assert all(torch.equal(p[k], q[k]) for k in ("blocks", "mask", "flag"))
        assert all(torch.equal(x[k], y[k]) for k in ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_q"))
