"""The LM head on CTA pairs at the edges of its tiles: rows of H around the
multiples of 32 and 256, vocabularies around 128 and 256 entries, hidden sizes
of an odd number of 64-column blocks (half a stage). Inputs are small integers,
so every product sum is exact in f32 (|sum| <= 4 * 5120 < 2^24) and the index
and the maximum are compared exactly, ties included (the first index wins)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dreams():
    import paper_2606_00535_gb300 as d
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    d._lib()
    return d


@pytest.mark.parametrize("rows,K,V", [
    (1, 64, 127), (31, 192, 128), (32, 64, 129), (33, 320, 255), (64, 128, 256), (65, 192, 257), (127, 64, 511),
    (128, 128, 513), (129, 448, 20000), (255, 64, 4097), (256, 192, 20001), (257, 128, 4096), (512, 320, 700),
    (513, 64, 33000), (1025, 192, 260), (2100, 64, 3000), (224, 5120, 300),
])
def test_tile_edges_and_ties_are_exact(dreams, rows, K, V):
    rng = np.random.default_rng(rows * 31 + K + V)
    h = rng.integers(-2, 3, (rows, K)).astype(np.float32)
    w = rng.integers(-2, 3, (V, K)).astype(np.float32)
    # equal entries across warps, CTAs and tiles: each maximum occurs more than once
    w[V // 2:] = w[:V - V // 2]
    h[rows // 2] = 0.0  # every entry ties at 0
    logits = h.astype(np.float64) @ w.astype(np.float64).T
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    hd, wd = torch.from_numpy(h).bfloat16().cuda(), torch.from_numpy(w).bfloat16().cuda()
    for _ in range(2):  # the second call finds its slots reset
        idx, mx = dreams.lm_head_argmax(hd, wd, want_max=True, status=st)
        np.testing.assert_array_equal(idx.cpu().numpy(), logits.argmax(1))
        np.testing.assert_array_equal(mx.cpu().numpy(), logits.max(1).astype(np.float32))
    assert int(st.item()) == 0


def test_infinities_and_nan(dreams):
    rows, K, V = 40, 64, 700
    h = torch.zeros((rows, K), dtype=torch.bfloat16)
    w = torch.zeros((V, K), dtype=torch.bfloat16)
    h[:, 0], h[1, 0], h[3, 0] = 1.0, -1.0, 0.0   # row 3: 0 * inf is NaN at the infinite entries
    w[:, 0] = -float("inf")
    w[300, 0] = w[301, 0] = float("inf")
    idx, mx = dreams.lm_head_argmax(h.cuda(), w.cuda(), want_max=True)
    idx, mx = idx.cpu(), mx.cpu()
    assert idx[0] == 300 and mx[0] == float("inf")
    assert idx[1] == 0 and mx[1] == float("inf")
    assert idx[3] == 0 and torch.isnan(mx[3])     # NaN is greatest, the first one wins
    assert idx[39] == 300
