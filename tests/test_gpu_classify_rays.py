"""Node classification in 3D with rays shared by a block's lines, against the oracle's winding number: bins from
far larger to smaller than a cell, and a box whose triangles' diagonals and edges lie exactly on rays (not
decided by the crossing count; the winding number of the mesh decides those cells)."""
import numpy as np
import pytest

from synth import Workload, small_workload
from tests.test_gpu_classify import _oracle_classes, _run
from tests.test_gpu_face_links import _box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,bins", [("sphere3", 1), ("sphere3", 5), ("bumpy3", 61), ("bumpy3", 150)])
def test_bin_sizes(kind, bins):
    w = small_workload(kind)
    g, res, solid, _ = _run(w, bins)
    rows = np.sort(np.random.default_rng(bins).choice(solid.shape[0], size=min(1500, solid.shape[0]), replace=False))
    want, band = _oracle_classes(w, res, rows)
    assert not ((solid[rows] != want) & ~band).any()
    g.close()


def test_rays_on_edges():
    h = 1.0 / 64
    t = _box(0.25 + h / 4, 0.75 + h / 4, 8)
    t[..., 1:] += np.float32(h / 4)  # y and z: the box's grid lines and diagonals pass through cell centres
    w = Workload("box", 3, t.reshape(-1, 3), np.arange(3 * t.shape[0], dtype=np.int32).reshape(-1, 3), root=8, n_levels=2,
                 bins=12, lattice=19)
    g, res, solid, undecided = _run(w)
    assert undecided > 0
    rows = np.arange(0, solid.shape[0], 3)
    want, band = _oracle_classes(w, res, rows)
    assert not ((solid[rows] != want) & ~band).any()
    g.close()
