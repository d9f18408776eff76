"""Rows that do not start on 16 bytes (a vocabulary with added tokens, a view
into a wider buffer). The argmax takes the values before a row's first 16-byte
boundary one by one and the others as aligned words; it must be the oracle's
at every offset of a row's start, with the maximum planted at the first, the
last and the boundary values. The draws must equal, bit for bit, those from
the same rows laid out on 16-byte boundaries. Lengths lie around the vectors,
the 256-value steps and the 1024-value segments."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dreams():
    import paper_2606_00535_gb300 as d
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    d._lib()
    return d


@pytest.mark.parametrize("V", [1, 7, 9, 255, 257, 1025, 5003])
@pytest.mark.parametrize("dtype,offset", [(torch.float32, o) for o in range(4)] + [(torch.bfloat16, o) for o in range(8)])
def test_unaligned_rows_equal_aligned_rows(dreams, dtype, offset, V):
    per = 16 // dtype.itemsize
    rows = 24
    rng = np.random.default_rng(V * 16 + offset)
    x = torch.from_numpy(2.0 * rng.standard_normal((rows, V), dtype=np.float32)).to(dtype)
    for r, at in enumerate((0, V - 1, min(V - 1, per - offset), min(V - 1, 8 * (V // 16)))):
        x[r, at] = 50.0
    x[5, V // 2] = float("-inf")
    x[6, V // 2] = float("inf")
    x[7, V // 2:] = float("nan")
    u = torch.from_numpy(rng.random(rows, dtype=np.float32)).cuda()
    pad = -(-V // per) * per
    aligned = torch.zeros((rows, pad), dtype=dtype, device="cuda")[:, :V]
    # a stride one past a multiple of 16 bytes: the rows' starts take every offset
    wide = torch.zeros((rows, pad + per + 1), dtype=dtype, device="cuda")[:, offset:offset + V]
    aligned.copy_(x)
    wide.copy_(x)
    assert torch.equal(dreams.vocab_sample(wide, 0.8, u), dreams.vocab_sample(aligned, 0.8, u))
    am = dreams.vocab_argmax(wide).cpu().numpy()
    ref = oracle.argmax(W.bits(x), bf16_bits=True) if dtype == torch.bfloat16 else oracle.argmax(x.numpy())
    np.testing.assert_array_equal(am, ref)


@pytest.mark.parametrize("V", [511, 512, 513, 519])
@pytest.mark.parametrize("dtype,offset", [(torch.float32, 3), (torch.bfloat16, 0), (torch.bfloat16, 5)])
def test_around_the_short_rows(dreams, dtype, offset, V):
    """Up to 512 values the argmax takes such a row value by value."""
    test_unaligned_rows_equal_aligned_rows(dreams, dtype, offset, V)
