"""Every kernel may start while the launch before it drains, and must wait for
it before it reads what that launch wrote. Here nothing is ready beforehand:
lengths, trees, uniforms, queries and logits are written by a torch kernel just
issued, over values that no call accepts or that would show, or by the
library's call before. A chain of all calls, issued back to back and replayed
from a captured graph, must give what it gives with the GPU waited for after
every launch."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dreams():
    import paper_2606_00535_gb300 as d
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    d._lib()
    return d


# 3 sequences: the attention is split and each CTA ranks its pairs, the tail takes several CTAs per sequence;
# 40: an ordering kernel runs ahead of the attention
@pytest.mark.parametrize("B,layers", [(3, 24), (40, 2)])
def test_calls_on_inputs_just_written(dreams, B, layers):
    rng = np.random.default_rng(B)
    T, V, Hq, Hkv, D, cap, mp, rounds = 12, 9000, 8, 2, 64, 2048, 5, 4
    f = lambda a: torch.as_tensor(a).cuda()  # noqa: E731
    bank = []
    for _ in range(rounds):
        par = np.stack([W.random_tree(rng, T) for _ in range(B)]).astype(np.int32)
        tok = rng.integers(0, V, (B, T)).astype(np.int32)
        x = rng.standard_normal((B, T, V)).astype(np.float32)
        for b in range(B):
            for i in range(T - 1, 0, -1):
                x[b, par[b, i], tok[b, i]] = 30.0 + T - i  # some drafts are accepted
        bank.append([f(a) for a in (par, tok, x, rng.random((2, B, T), dtype=np.float32))] +
                    [W.bf16(rng.standard_normal(n)).cuda() for n in ((B, T, Hq, D), (B * T, 128), (B, 2, 8, 500))])
    k0, v0 = (W.bf16(rng.standard_normal((layers, B, cap, Hkv, D), dtype=np.float32)).cuda() for _ in range(2))
    kl0, full = f(rng.integers(900, 1700, B).astype(np.int32)), torch.full((B,), T, dtype=torch.int32, device="cuda")
    kv = dreams.KVCache(k0.clone(), v0.clone())
    i32 = lambda *s: torch.zeros(s, dtype=torch.int32, device="cuda")  # noqa: E731
    par, tok, tl, lens = i32(B, T), i32(B, T), i32(B), [i32(B) for _ in range(4)]
    trees = [dreams.Tree(par, tok, tl, n) for n in lens]  # call n's new lengths are call n + 1's lengths
    outs = [(i32(B), i32(B, mp), i32(B, mp), n) for n in lens[1:]]
    logits, drf = torch.zeros((B, T, V), device="cuda"), torch.zeros((B, T, V), device="cuda")
    u, q, status, pred = torch.zeros((2, B, T), device="cuda"), torch.empty_like(bank[0][4]), i32(1), i32(B, T)
    att, att2 = torch.empty_like(q), torch.empty((B, mp, Hq, D), dtype=torch.bfloat16, device="cuda")
    q2 = torch.empty_like(att2)
    lse = torch.zeros((B, T, Hq), device="cuda")
    hid, vis = torch.empty_like(bank[0][5]), torch.empty_like(bank[0][6])
    head = W.bf16(rng.standard_normal((V, 128))).cuda()
    am, top, best, imp, keep_i = i32(B, T), i32(B * T), lse.new_zeros(B * T), lse.new_zeros((B, 400)), i32(B, 90)
    results = (*outs[0], *outs[1], *outs[2], att, lse, att2, pred, am, top, best, imp, keep_i)
    kept = [[torch.zeros_like(t) for t in results] for _ in range(rounds)]

    def chain(wait):
        for t, v in ((kv.k, k0), (kv.v, v0), (lens[3], kl0)):
            t.copy_(v)
        for (par_r, tok_r, x_r, u_r, q_r, hid_r, vis_r), keep in zip(bank, kept):
            steps = [
                lambda: (lens[0].copy_(lens[3]), par.fill_(-9), tl.fill_(-3), q.fill_(float("nan"))),
                lambda: (par.copy_(par_r), tok.copy_(tok_r), q.copy_(q_r), tl.copy_(full)),
                lambda: dreams.tree_verify_attn(q, kv, trees[0], 0.125, out=att, lse=lse, status=status),
                lambda: (logits.fill_(float("nan")), logits.copy_(x_r)),
                lambda: dreams.vocab_argmax(logits, out=am),
                lambda: dreams.verify_step(logits, trees[0], kv, mp, outputs=outs[0], status=status),
                lambda: dreams.kv_compact(kv, lens[0], outs[0][0], outs[0][1], status=status),
                lambda: (u.fill_(1.0), u.copy_(u_r)),
                lambda: dreams.verify_step_sampled(logits, trees[1], kv, mp, 2.0, u[0], sample_out=pred,
                                                   outputs=outs[1], status=status),
                lambda: (drf.copy_(logits), drf.mul_(0.7), u.mul_(0.9)),
                lambda: dreams.verify_step_speculative(logits, drf, trees[2], kv, mp, 2.0, u[0], u[1], outputs=outs[2],
                                                       status=status),
                lambda: (att2.fill_(7.0), q2.fill_(float("nan")), q2.copy_(att[:, :mp])),
                # as many queries as the walk before accepted, behind its new lengths
                lambda: dreams.attention(q2, kv, outs[2][0], lens[3], 0.125, dreams.ATTN_CAUSAL, out=att2,
                                         status=status),
                lambda: (hid.fill_(float("nan")), hid.copy_(hid_r)),
                lambda: dreams.lm_head_argmax(hid, head, out=top, out_max=best, status=status),
                lambda: (vis.fill_(float("nan")), vis.copy_(vis_r)),
                lambda: [a.copy_(t) for a, t in zip((imp, keep_i), dreams.visual_importance(vis, 60, 400, 90))],
                lambda: [a.copy_(t) for a, t in zip(keep, results)],
            ]
            for step in steps:
                step()
                if wait:
                    torch.cuda.synchronize()
        return [t for keep in kept for t in keep] + [kv.k, kv.v]

    want = [t.clone() for t in chain(True)]
    assert int(status.item()) == 0 and (torch.stack([want[len(results) * r] for r in range(rounds)]) > 1).any()

    def check():
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        for n, (a, w) in enumerate(zip([t for keep in kept for t in keep] + [kv.k, kv.v], want)):
            assert torch.equal(a, w), n

    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for _ in range(5):
            chain(False)
            check()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            chain(False)
        for _ in range(5):
            for keep in kept:
                for t in keep:
                    t.zero_()
            graph.replay()
            check()
