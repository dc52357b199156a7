"""Face sums of the q adjoint (a tile's links grouped by face in shared memory, integer sums over the
tiles) against FP64 from the same links: faces that fill whole tiles, tiles of hundreds of faces, a part
tile, and weights of very different size, zero and non-finite.

Tolerance per face, from the arithmetic: a link's FP32 term grad_q w, w = (v0 - x - t d) / (d . n), carries a
few roundings of vectors no larger than R + 2 h (R the face's extent) and of the quotient, so it is within
16 u |grad_q / (d . n)| (R + 2 h) of its value (u = 2^-24); the edges multiply it by at most E = 2 R, and the
corner that holds n S adds 16 u |n| |grad_q / (d . n)|."""
import numpy as np
import pytest

from synth import Workload
from synth import geometry as G
from tests import gpu_util as U

pytestmark = pytest.mark.gpu

DIRS2 = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]], float)
DIRS3 = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0],
                  [-1, -1, 0], [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1],
                  [0, -1, -1], [0, 1, -1], [0, -1, 1]], float)


def _mesh(kind):
    if kind == "big_faces":  # thousands of links per face: a tile has one or two faces
        v, f = G.jittered_sphere(0, radius=0.3, centre=(0.5, 0.49, 0.51), sigma=1e-4, seed=3)
        return Workload(kind, 3, v, f, root=8, n_levels=4, bins=4, lattice=19)
    if kind == "small_faces":  # about one link per face: a tile has hundreds of faces
        v, f = G.jittered_sphere(5, radius=0.3, centre=(0.5, 0.49, 0.51), sigma=1e-5, seed=4)
        return Workload(kind, 3, v, f, root=6, n_levels=2, bins=24, lattice=19)
    if kind == "segments":
        v, f = G.circle_polygon(91, 0.313, (0.47, 0.52))
        return Workload(kind, 2, v, f, root=10, n_levels=4, bins=7, lattice=9)
    raise KeyError(kind)


def _reference(w, V, q, faces, dirs, cells, gq):
    """Per face in FP64: gradient [F, D, D] and the tolerance [F]."""
    D, h = w.dim, 1.0 / (4 * w.root * 2 ** (w.n_levels - 1))
    P = V.astype(np.float64)[faces]
    d = (DIRS2 if D == 2 else DIRS3)[dirs] * h
    x = (cells + 0.5) * h
    e1 = P[:, 1] - P[:, 0]
    if D == 3:
        e2 = P[:, 2] - P[:, 0]
        n = np.cross(e1, e2)
    else:
        n = np.stack([e1[:, 1], -e1[:, 0]], 1)
    den = (d * n).sum(1)
    wv = (P[:, 0] - x - q[:, None] * d) / den[:, None]
    if D == 3:
        g1, g2 = np.cross(e2, wv), np.cross(wv, e1)
        g = np.stack([n / den[:, None] - g1 - g2, g1, g2], 1)
    else:
        g1 = np.stack([-wv[:, 1], wv[:, 0]], 1)
        g = np.stack([n / den[:, None] - g1, g1], 1)
    F = V.shape[0]
    out, tol = np.zeros((F, D, D)), np.zeros(F)
    np.add.at(out, faces, gq[:, None, None] * g)
    R = np.abs(P - P[:, :1]).max((1, 2))
    np.add.at(tol, faces, 16 * 2.0 ** -24 * np.abs(gq / den) * (6 * R * (R + 2 * h) + np.abs(n).max(1)))
    return out, tol


@pytest.mark.parametrize("kind", ["big_faces", "small_faces", "segments"])
def test_face_sums(kind):
    import torch

    from paper_2502_16310_gb300 import AmrGeom

    w = _mesh(kind)
    V = w.verts[w.idx]
    g = AmrGeom(w.dim, (w.root,) * w.dim)
    g.load(torch.from_numpy(np.ascontiguousarray(V)).cuda())
    g.bin(w.bins)
    r = g.refine(w.n_levels, 0.0, 1.0, w.lattice, True, True)
    q = U.to_np(r["link_q"]).astype(np.float64)
    faces = U.to_np(r["link_face"], np.uint32).astype(np.int64)
    dirs = U.to_np(r["link_dir"]).astype(np.int64)
    nc = 64 if w.dim == 3 else 16
    ids = U.to_np(r["adj_cell"], np.uint32)[U.to_np(r["link_cell"], np.uint32).astype(np.int64)].astype(np.int64)
    blocks = U.to_np(r["levels"][-1]["blocks"]).copy()
    cells = np.stack([4 * blocks[ids // nc, a] + ((ids % nc) >> (2 * a)) % 4 for a in range(w.dim)], 1).astype(float)
    nl = q.size
    assert nl % 256 != 0
    per_tile = [np.unique(faces[i:i + 256]).size for i in range(0, nl, 256)]
    assert {"big_faces": min(per_tile) <= 2, "small_faces": max(per_tile) > 100, "segments": nl > 1024}[kind]
    rng = np.random.default_rng(7)
    plain = rng.normal(size=nl)
    for gq in (plain, plain * 10.0 ** rng.uniform(-30, 28, size=V.shape[0])[faces], plain * (faces % 3 == 0)):
        gq = gq.astype(np.float32)
        ref, tol = _reference(w, V, q, faces, dirs, cells, gq.astype(np.float64))
        dev = torch.from_numpy(gq).cuda()
        got = g.q_backward(dev)
        again = g.q_backward(dev)
        assert torch.equal(got, again)
        got = got.cpu().numpy().astype(np.float64)
        err = np.abs(got - ref).max((1, 2))
        bad = err > tol + 2.0 ** -23 * np.abs(ref).max((1, 2)) + 1e-37
        assert not bad.any(), (int(bad.sum()), float((err[bad] / tol[bad]).max()))
        assert (got[tol == 0] == 0).all()
    gq = plain.astype(np.float32)
    gq[nl // 2] = np.inf
    got = g.q_backward(torch.from_numpy(gq).cuda()).cpu().numpy()
    hit = np.zeros(V.shape[0], bool)
    hit[faces[nl // 2]] = True
    assert np.isnan(got[hit]).all() and np.isfinite(got[~hit]).all()
    g.close()
