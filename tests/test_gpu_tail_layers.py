"""GPU parity of the verification tail on many-layer caches, where the walk
launch spreads each sequence's compaction over several CTAs: cache columns
(16-byte units of all layers, K and V, all heads) just below, at and above one
CTA's 256, an odd count, and a whole model's worth; predictions in the
workspace (cleared by the last CTA to read them) and in the caller's array.
Every result is exact: predictions, walk, and every byte of every layer. A
decode loop may also advance its lengths in place (new_kv_len is kv_len), which
must change nothing."""
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


# columns = 2 * layers * Hkv * D / 8
@pytest.mark.parametrize("layers,Hkv,D,paged", [(1, 8, 120, False), (1, 8, 128, True), (1, 9, 128, False),
                                                (3, 5, 72, True), (24, 16, 128, False)])
@pytest.mark.parametrize("own_pred", [False, True])
def test_tail_compacts_every_layer(dreams, layers, Hkv, D, paged, own_pred):
    rng = np.random.default_rng(layers * 100 + Hkv)
    B, T, V, cap = 4, 21, 300, 128
    tl = np.array([21, 1, 9, 0], np.int32)  # the last one is invalid
    kl = np.array([100, 40, 60, 5], np.int32)
    par = np.full((B, T), -1, np.int32)
    for b in range(B):
        if tl[b]:
            par[b, :tl[b]] = W.random_tree(rng, int(tl[b]))
    tok = rng.integers(0, V, (B, T)).astype(np.int32)
    x = rng.standard_normal((B, T, V)).astype(np.float32)
    for b in range(B):  # each node predicts the child with the deepest subtree: long accepted paths
        height = np.zeros(T, int)
        for i in range(int(tl[b]) - 1, 0, -1):
            height[par[b, i]] = max(height[par[b, i]], height[i] + 1)
            x[b, par[b, i], tok[b, i]] = 50.0 + height[i]
    pred = oracle.argmax(x.reshape(-1, V)).reshape(B, T)
    ref = oracle.accept_path(pred, par, tok, tl, kl, T + 1)
    assert ref["accept_len"][0] > 2
    if paged:
        table = rng.permutation(2 * B).astype(np.int32).reshape(B, 2)
        lay = oracle.KVLayout(cap, Hkv, D, page_table=table, page_size=64, num_pages=2 * B)
        shape = (layers, 2 * B, 64, Hkv, D)
    else:
        lay = oracle.KVLayout(cap, Hkv, D)
        shape = (layers, B, cap, Hkv, D)
    k, v = (W.bf16(rng.standard_normal(shape, dtype=np.float32)) for _ in range(2))
    kv = dreams.KVCache(k.cuda(), v.cuda(), torch.from_numpy(table).cuda() if paged else None)
    f = lambda a: torch.as_tensor(a).cuda()  # noqa: E731
    tree = dreams.Tree(f(par), f(tok), f(tl), f(kl))
    ws = torch.zeros(dreams.verify_step_workspace_size(tree, V), dtype=torch.uint8, device="cuda")
    am = torch.full((B, T), -7, dtype=torch.int32, device="cuda") if own_pred else None
    ko, vo = W.bits(k).copy(), W.bits(v).copy()
    for _ in range(2):  # the second call on the same, again zero-filled, workspace
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        r = dreams.verify_step(f(x), tree, kv, T + 1, argmax_out=am, workspace=ws, status=st)
        torch.cuda.synchronize()
        assert int(st.item()) == dreams.DATA_BAD_TREE_LEN
        assert int(ws.count_nonzero().item()) == 0
        for key in ("accept_len", "path", "out_tokens", "new_kv_len"):
            np.testing.assert_array_equal(r[key].cpu().numpy(), ref[key], err_msg=key)
        for n in range(layers):
            ko[n], vo[n], ost = oracle.kv_compact(ko[n], vo[n], lay, kl, ref["accept_len"], ref["path"])
            assert ost == 0
        assert np.array_equal(W.bits(kv.k.cpu()), ko) and np.array_equal(W.bits(kv.v.cpu()), vo)


@pytest.mark.parametrize("layers,B,T,V", [(32, 16, 64, 600), (4, 3, 9, 5000)])
@pytest.mark.parametrize("call", ["greedy", "greedy_own", "sampled", "speculative"])
def test_lengths_advance_in_place(dreams, call, layers, B, T, V):
    """Calls in a row on one cache, each on the lengths that the call before
    wrote over its own. With 32 layers, 16 sequences and 64 rows each, 512 CTAs
    of the walk start as the 1024 of the rows leave the SMs."""
    rng = np.random.default_rng(layers + T)
    Hkv, D, cap, steps = 8, 128, 160, 6
    f = lambda a: torch.as_tensor(a).cuda()  # noqa: E731
    kl0 = rng.integers(0, 64, B).astype(np.int32)
    tl = rng.integers(max(1, T - 20), T + 1, B).astype(np.int32)
    par = np.full((B, T), -1, np.int32)
    for b in range(B):
        par[b, :tl[b]] = W.random_tree(rng, int(tl[b]))
    tok = rng.integers(0, V, (B, T)).astype(np.int32)
    x = rng.standard_normal((B, T, V)).astype(np.float32)
    np.put_along_axis(x, x.argmax(-1)[..., None], 20.0, -1)
    for b in range(B):  # every node's first child is its prediction
        for i in range(int(tl[b]) - 1, 0, -1):
            x[b, par[b, i], tok[b, i]] = 50.0 + (int(tl[b]) - i)
    u_np, zero = rng.random((B, T), dtype=np.float32), np.zeros((B, T), np.float32)
    logits, u, u0 = f(x), f(u_np), f(zero)
    pred = oracle.argmax(x.reshape(-1, V)).reshape(B, T)
    lay = oracle.KVLayout(cap, Hkv, D)
    ko, vo = (rng.integers(0, 1 << 16, (layers, B, cap, Hkv, D), np.uint16) for _ in range(2))
    kv = dreams.KVCache(*(f(a.view(np.int16)).view(torch.bfloat16) for a in (ko, vo)))
    tree = dreams.Tree(f(par), f(tok), f(tl), f(kl0))
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    acc, path, toks = (torch.empty(s, dtype=torch.int32, device="cuda") for s in ((B,), (B, 4), (B, 4)))
    am = torch.empty((B, T), dtype=torch.int32, device="cuda") if call == "greedy_own" else None
    for _ in range(steps):
        out = (acc, path, toks, tree.kv_len)
        if call == "sampled":  # at this temperature the draws are the argmax
            dreams.verify_step_sampled(logits, tree, kv, 4, 1e-3, u, outputs=out, status=st)
        elif call == "speculative":  # draft == target and uniforms of 0: first children are accepted
            dreams.verify_step_speculative(logits, logits, tree, kv, 4, 1e-3, u0, u, outputs=out, status=st)
        else:
            dreams.verify_step(logits, tree, kv, 4, argmax_out=am, outputs=out, status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    kl = kl0
    for _ in range(steps):
        ref = (oracle.spec_path(x, x, par, tok, tl, kl, 4, 1e-3, zero, u_np) if call == "speculative" else
               oracle.accept_path(pred, par, tok, tl, kl, 4))
        for n in range(layers):
            ko[n], vo[n], ost = oracle.kv_compact(ko[n], vo[n], lay, kl, ref["accept_len"], ref["path"])
            assert ost == 0
        kl = ref["new_kv_len"]
    assert (kl > kl0 + steps).any()
    np.testing.assert_array_equal(tree.kv_len.cpu().numpy(), kl)
    np.testing.assert_array_equal(path.cpu().numpy(), ref["path"])
    np.testing.assert_array_equal(toks.cpu().numpy(), ref["out_tokens"])
    assert np.array_equal(W.bits(kv.k.cpu()), ko) and np.array_equal(W.bits(kv.v.cpu()), vo)
