"""Point predicate, mark-only walks: which calls gather their faces (they build the entries' spheres first), on both
sides of the rule: small faces in few bins do; few, wide or many-binned faces are taken one at a time.  The marks
are those of the walk that keeps every pair."""
import numpy as np
import pytest

from tests.test_gpu_face_pass import OFF

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("freq,B,d,gathers", [(30, 8, 0.05, True), (30, 48, 0.05, False), (2, 8, 0.05, False),
                                              (10, 4, 0.12, True), (4, 2, 0.004, False)])
def test_gathering(freq, B, d, gathers):
    import torch

    from paper_2502_16310_gb300 import AmrGeom
    from synth import geometry as G

    v, f = G.geodesic_sphere_unit(freq)
    v = torch.from_numpy((0.5 + 0.31 * v).astype(np.float32)).cuda()
    f = torch.from_numpy(f.astype(np.int32)).cuda()
    out = []
    for adjacency in (False, True):
        g = AmrGeom(3, (4,) * 3)
        g.load(v, f)
        g.bin(B)
        g.timing(True)
        r = g.refine(1, d, 0.0, 0, adjacency, False, predicate=1, face_pass=OFF)
        torch.cuda.synchronize()
        out.append(r["levels"][0]["mask"].clone())
        if not adjacency:
            assert ("entry_spheres" in g.timings()) == gathers
        g.close()
    assert torch.equal(*out) and int((out[0] != 0).sum()) > 0
