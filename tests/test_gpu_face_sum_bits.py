"""Face sums of the q adjoint keep a small link beside large ones that cancel: on dyadic planes every term is exact in
FP32, a pair of opposite links on one line cancels exactly, and what is left of the face is a link whose weight is
2^-40 of theirs.  The sums are fixed point with a spacing of 2^-(62 - b) of a bound that lies within 2^5 of the
largest term (a factor 4 from the exponents' sum, up to 8 from twice the extent to its power of two), b the bits of
the face's number of links (at most 11 for a triangle of 8 cells): an error of 2^-46 of the largest term at most, in
a mesh of over a million links."""
import numpy as np
import pytest

from tests import gpu_util as U
from tests.test_gpu_face_sums import DIRS3

pytestmark = pytest.mark.gpu


def test_small_links_beside_cancelling_ones():
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    h, root, levels = 1.0 / 128, 16, 2
    g = np.arange(16, 112, 8) * h
    a, b = np.meshgrid(g, g, indexing="ij")
    quad = np.stack([np.stack(c, -1) for c in ((a, b), (a + 8 * h, b), (a + 8 * h, b + 8 * h), (a, b + 8 * h))], -2)
    quad = quad.reshape(-1, 4, 2)
    tris = []
    for k in range(20, 108, 6):  # a quarter of a cell above the centres of layer k
        q = np.concatenate([quad, np.full(quad.shape[:2] + (1,), (k + 0.75) * h)], -1)
        tris += [q[:, [0, 1, 2]], q[:, [0, 2, 3]]]
    V = np.concatenate(tris)
    ctx = AmrGeom(3, (root,) * 3)
    ctx.load(torch.from_numpy(V.astype(np.float32)).cuda())
    ctx.bin(32)
    r = ctx.refine(levels, 0.0, 1.0, 19, True, True)
    q = U.to_np(r["link_q"]).astype(np.float64)
    face = U.to_np(r["link_face"], np.uint32).astype(np.int64)
    dirs = U.to_np(r["link_dir"]).astype(np.int64)
    ids = U.to_np(r["adj_cell"], np.uint32)[U.to_np(r["link_cell"], np.uint32).astype(np.int64)].astype(np.int64)
    blocks = U.to_np(r["levels"][-1]["blocks"]).copy()
    cell = np.stack([4 * blocks[ids // 64, c] + ((ids % 64) >> (2 * c)) % 4 for c in range(3)], 1)
    assert q.size > 1 << 20
    back = {(tuple(c), d): i for i, (c, d) in enumerate(zip(cell, dirs)) if face[i] % 97 == 0}
    gq, used = np.zeros(q.size, np.float32), {}
    for (c, d), i in back.items():
        f = face[i]
        ahead = tuple(int(x) for x in np.array(c) + DIRS3[d].astype(int))
        j = back.get((ahead, d + 1)) if d % 2 else None  # directions 2 l + 1 and 2 l + 2 are opposite
        if j is not None and face[j] == f and used.setdefault(f, 0) < 9:
            gq[i] = gq[j] = 1.0
            used[f] += 1
    small = {}
    for (c, d), i in back.items():
        if gq[i] == 0 and face[i] in used and face[i] not in small:
            gq[i] = 2.0 ** -40
            small[face[i]] = i
    assert len(small) > 20 and min(used[f] for f in small) > 2
    got = ctx.q_backward(torch.from_numpy(gq).cuda()).cpu().numpy().astype(np.float64)
    ctx.close()
    e1, e2 = V[:, 1] - V[:, 0], V[:, 2] - V[:, 0]
    n = np.cross(e1, e2)
    for f, i in small.items():
        d = DIRS3[dirs[i]] * h
        x = (cell[i] + 0.5) * h
        w = (V[f, 0] - x - q[i] * d) / (d @ n[f])
        g1, g2 = np.cross(e2[f], w), np.cross(w, e1[f])
        want = 2.0 ** -40 * np.stack([n[f] / (d @ n[f]) - g1 - g2, g1, g2])
        largest = np.abs(n[f]).max() / np.abs(n[f] @ np.array([0, 0, h]))  # of a link with weight 1
        assert np.abs(got[f] - want).max() <= 4 * 2.0 ** -46 * largest, f
        assert np.abs(want).max() > 2.0 ** -43 * largest
