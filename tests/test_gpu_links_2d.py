"""D2Q9 links where the FP32 filter meets its bounds: segments whose ends lie on cell centres and link ends,
parallel to lattice directions, far shorter and far longer than a cell, against the FP64 oracle."""
import numpy as np
import pytest

from oracle.oracle import Domain, OracleGeometry
from synth import Workload
from tests import gpu_util as U
from tests.test_gpu_mark_cells import _soup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("root", [4, 5])
@pytest.mark.parametrize("size,snap", [(0.0005, None), (0.03, None), (0.3, None), (0.03, 1 / 64), (0.1, 1 / 80)])
def test_links_2d_against_oracle(root, size, snap):
    v, f = _soup(2, size, 60, seed=int(1e4 * size) + root, snap=snap)
    w = Workload("soup", 2, v, f, root=root, n_levels=2, bins=6, lattice=9)
    out = U.run_gpu(w)
    fin = out["levels"][-1]
    geo = OracleGeometry(2, v, f)
    geo.bin(Domain.unit(2, root), 6)
    U.compare_links(geo, 2, 1, 9, fin["blocks"], out["adj_cell"], out["link_cell"],
                    out["link_dir"], out["link_q"], out["link_face"], sample=150, rng=np.random.default_rng(3))
    assert out["link_q"].shape[0] > 0
