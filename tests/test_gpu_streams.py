"""GPU parity of calls on a stream that is not the current one, which is kept
busy meanwhile, with the allocator's memory dirtied beforehand: the kept
workspaces of the argmax, the verification step and the LM head, whose slots
and counters must be zero, are created small, grown and used on that stream."""
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


def test_calls_on_another_stream(dreams):
    rng = np.random.default_rng(1)
    side = torch.cuda.Stream()
    f = lambda a: torch.as_tensor(a).cuda()  # noqa: E731
    for B, T, V in ((1, 3, 9000), (2, 20, 40000), (8, 60, 20000)):  # rows split over CTAs, growing
        par = np.stack([W.random_tree(rng, T) for _ in range(B)]).astype(np.int32)
        tok = rng.integers(0, V, (B, T)).astype(np.int32)
        tl, kl = np.full(B, T, np.int32), rng.integers(0, 30, B).astype(np.int32)
        x = rng.standard_normal((B, T, V)).astype(np.float32)
        h, w = W.bf16(rng.standard_normal((B * T, 128))), W.bf16(rng.standard_normal((V, 128)))
        pred = oracle.argmax(x.reshape(-1, V)).reshape(B, T)
        ref = oracle.accept_path(pred, par, tok, tl, kl, 5)
        k = torch.zeros((B, 128, 1, 64), dtype=torch.bfloat16, device="cuda")
        logits, hg, wg = f(x), h.cuda(), w.cuda()
        kv, tree = dreams.KVCache(k, k.clone()), dreams.Tree(f(par), f(tok), f(tl), f(kl))
        want = dreams.lm_head_argmax(hg, wg)  # on the current stream
        outs = tuple(torch.empty(s, dtype=torch.int32, device="cuda") for s in ((B,), (B, 5), (B, 5), (B,)))
        am, am2 = (torch.empty((B, T), dtype=torch.int32, device="cuda") for _ in range(2))
        got = torch.empty(B * T, dtype=torch.int32, device="cuda")
        dirt = [torch.full((1 << n,), 0x55, dtype=torch.uint8, device="cuda") for n in range(9, 21)]
        with torch.cuda.stream(side):
            dirt += [torch.full((1 << n,), 0x55, dtype=torch.uint8, device="cuda") for n in range(9, 21)]
        torch.cuda.synchronize()
        del dirt
        torch.cuda._sleep(20_000_000)  # the current stream is busy for about 10 ms
        dreams.vocab_argmax(logits, out=am, stream=side)
        dreams.verify_step(logits, tree, kv, 5, argmax_out=am2, outputs=outs, stream=side)
        dreams.lm_head_argmax(hg, wg, out=got, stream=side)
        side.synchronize()
        assert np.array_equal(am.cpu().numpy(), pred) and np.array_equal(am2.cpu().numpy(), pred)
        for t, key in zip(outs, ("accept_len", "path", "out_tokens", "new_kv_len")):
            np.testing.assert_array_equal(t.cpu().numpy(), ref[key], err_msg=key)
        assert torch.equal(got, want)
