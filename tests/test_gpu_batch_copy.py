"""amr_batch_copy (one launch for a batch geometry's arrays) against tensor operations: lengths about a tile's
edges, sources at any element offset, more arrays than one launch takes, indices that wrap; bad calls refused."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rows(copies):
    return np.array([(s.data_ptr(), d.data_ptr(), s.numel(), m, k) for s, d, m, k in copies], dtype=np.int64)


@pytest.mark.parametrize("lengths", [[1], [4095, 4096, 4097, 0, 3], list(range(1, 34)), [100_003] * 5])
def test_copies_equal_tensor_operations(lengths):
    import torch

    from paper_2502_16310_gb300 import AmrBatch, binding as B

    g = torch.Generator(device="cuda").manual_seed(len(lengths))
    copies, want = [], []
    for i, n in enumerate(lengths):
        raw = torch.randint(-2**31, 2**31 - 1, (2 * n + 8,), generator=g, device="cuda", dtype=torch.int64)
        w32 = raw.to(torch.int32)[i % 4:i % 4 + n]
        w8 = raw.to(torch.uint8)[i % 7:i % 7 + n]
        minus = 12345 * i - 7
        for src, dtype, m, kind, ref in [
                (w8, torch.uint8, 0, B.AMR_COPY_8, w8), (w32, torch.int32, 0, B.AMR_COPY_32, w32),
                (raw[1:1 + n], torch.int64, 0, B.AMR_COPY_64, raw[1:1 + n]),
                (w32, torch.int32, minus, B.AMR_COPY_I32, w32 - minus),
                (w32, torch.int64, minus, B.AMR_COPY_I32_I64, w32.long() - minus)]:
            copies.append((src, torch.full((n,), 77, dtype=dtype, device="cuda"), m, kind))
            want.append(ref)
    b = AmrBatch(2)
    rows = _rows(copies)
    assert B.lib().amr_batch_copy(b.b, rows.ctypes.data, len(copies), torch.cuda.current_stream().cuda_stream) == 0
    for (_, got, _, _), ref in zip(copies, want):
        assert torch.equal(got, ref)


def test_bad_calls_are_refused():
    import torch

    from paper_2502_16310_gb300 import AmrBatch, binding as B

    b = AmrBatch(2)
    t = torch.zeros(4, dtype=torch.int32, device="cuda")
    good = _rows([(t, t.clone(), 0, B.AMR_COPY_32)])
    for col, bad in [(4, 3), (2, -1), (0, 0), (1, 0)]:
        rows = good.copy()
        rows[0, col] = bad
        assert B.lib().amr_batch_copy(b.b, rows.ctypes.data, 1, None) == B.AMR_EINVAL
    assert B.lib().amr_batch_copy(b.b, None, 1, None) == B.AMR_EINVAL
    assert B.lib().amr_batch_copy(b.b, good.ctypes.data, 0, None) == 0
