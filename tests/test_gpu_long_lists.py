"""Adjacency lists of blocks with few, many and more survivor records than are kept or sorted (64 staged,
1,024 kept): a cluster of faces beside a few blocks, against the FP64 oracle and the face-by-face levels."""
import numpy as np
import pytest

from synth import Workload
from tests.test_gpu_point import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n", [64, 65, 250, 1024, 1500])
def test_long_lists_against_oracle(dim, n):
    rng = np.random.default_rng(n + dim)
    v = (rng.uniform(0.42, 0.46, (n, 1, dim)) + rng.uniform(-0.003, 0.003, (n, dim, dim))).astype(np.float32)
    f = rng.permutation(n * dim).astype(np.int32).reshape(n, dim)
    v = v.reshape(-1, dim)[np.argsort(f.reshape(-1))]
    w = Workload("cluster", dim, v, f, root=4, n_levels=2, bins=5, lattice=9 if dim == 2 else 19)
    out = _check(w, 0.0625, sample=6)
    counts = np.diff(out["adj_off"][:out["adj_cell"].shape[0] + 1].astype(np.int64))
    assert counts.max() > 0.9 * n
