"""Point predicate where the quick test (a sphere about each face's centroid) meets the general one: faces
from far below d to larger than a block, corners free or on cell and block planes (distances that are exactly
d), across the domain's sides; masks, lists and links against the FP64 oracle outside its 1e-6 h band."""
import pytest

from synth import Workload
from tests.test_gpu_mark_cells import _soup
from tests.test_gpu_point import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("d", [0.0625, 0.2])
@pytest.mark.parametrize("size,snap", [(0.002, None), (0.08, None), (0.4, None), (0.08, 1 / 64)])
def test_quick_test_against_oracle(dim, d, size, snap):
    v, f = _soup(dim, size, 24, seed=int(1000 * size) + dim, snap=snap)
    out = _check(Workload("soup", dim, v, f, root=4, n_levels=2, bins=5, lattice=9 if dim == 2 else 19), d, sample=40)
    assert out["adj_cell"].shape[0] > 0
