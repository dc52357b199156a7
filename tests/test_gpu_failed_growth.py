"""A device allocation that fails inside a call leaves a context whose next calls work: each allocation of a call
fails once, then the same call is made again, and its outputs are those of a context that never failed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


KEYS = ("adj_cell", "adj_off", "adj_ids", "link_cell", "link_dir", "link_q", "link_face")


def _mesh(kind):
    """cluster: more records than a block's usual share; wide: more links than a quarter above the pairs."""
    if kind == "cluster":
        rng = np.random.default_rng(3)
        return (rng.uniform(0.42, 0.46, (900, 1, 3)) + rng.uniform(-0.003, 0.003, (900, 3, 3))).astype(np.float32), 2
    z = 0.5 + 0.37 / 128
    return np.array([[[0.1, 0.1, z], [0.9, 0.1, z], [0.9, 0.9, z]], [[0.1, 0.1, z], [0.9, 0.9, z], [0.1, 0.9, z]]],
                    np.float32), 16


def _each_fails_once(kind, call):
    """call(g, mesh) -> tensors, with every one of its device allocations failing in turn."""
    import torch

    from paper_2502_16310_gb300 import AmrError, AmrGeom
    from paper_2502_16310_gb300 import binding as Bd

    mesh, root = _mesh(kind)
    dev = torch.from_numpy(mesh).cuda()
    live, state = {}, {"n": 0, "fail": -1}

    @Bd.DEV_ALLOC
    def alloc(n, user):
        state["n"] += 1
        if state["n"] - 1 == state["fail"]:
            return None
        t = torch.empty(int(n), dtype=torch.uint8, device="cuda")
        live[t.data_ptr()] = t
        return t.data_ptr()

    @Bd.DEV_FREE
    def free(p, user):
        torch.cuda.synchronize()
        del live[p]

    def context(fail):
        state["fail"] = -1
        g = AmrGeom(3, (root,) * 3, dev_alloc=alloc, dev_free=free)
        state["n"], state["fail"] = 0, fail
        return g

    g = context(-1)
    want = call(g, dev)
    total = state["n"]
    g.close()
    assert total > 5
    for fail in range(total):
        g = context(fail)
        with pytest.raises(AmrError) as e:
            call(g, dev)
        assert e.value.status == Bd.AMR_ENOMEM
        for _ in range(2):
            for a, b in zip(call(g, dev), want):
                assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), fail
        g.close()
    assert not live


@pytest.mark.parametrize("kind", ["cluster", "wide"])
def test_binning(kind):
    import torch

    def call(g, dev):
        g.load(dev)
        b = g.bin(8)
        torch.cuda.synchronize()
        bins = torch.bucketize(torch.arange(b["nnz"], device="cuda"), b["offsets"][1:].long(), right=True)
        return [b["offsets"].clone(), torch.sort(bins * (1 << 29) + b["ids"].long())[0]]

    _each_fails_once(kind, call)


@pytest.mark.parametrize("kind", ["cluster", "wide"])
def test_refinement(kind):
    import torch

    def call(g, dev):
        g.load(dev)
        g.bin(8)
        r = g.refine(2, 0.0, 1.0, 19, True, True, face_pass=2)
        torch.cuda.synchronize()
        return [lv["mask"].clone() for lv in r["levels"]] + [r[k].clone() for k in KEYS]

    _each_fails_once(kind, call)
