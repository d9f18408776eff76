"""Performance cases of the tree-verification library.

Each case is one call (or the two calls of one decoding step) of the package's
public entry points on inputs shaped like the decoding this library serves: the
target model's verification of a draft tree for one user or for a batch of
users, the prefill before it, and the draft model's visual-token selection.

`listed()` is the fixed set; `draw()` gives further cases of the same ranges.
`prepare()` makes what a serving program holds before the call (inputs, KV
cache, output buffers), `run()` makes the call, `exact()` restates the results
in 64-bit torch without the library.
"""
import math

import numpy as np
import torch

import paper_2606_00535_gb300 as dreams

DEV = "cuda"
PAGE = 64

ATTN, VERIFY, SAMPLED, SPECULATIVE = "tree_attention", "verify", "verify_sampled", "verify_speculative"
STEP, MODES, LM_HEAD, IMPORTANCE = "step", "attention", "lm_head", "importance"


def listed():
    return [
        # The smallest step: attention and verification of a 16-node tree on a
        # short prompt. Launches and latency are all there is.
        dict(name="step_tiny", kind=STEP, B=1, T=16, depth=4, Hq=4, Hkv=4, D=64, L=256, ragged=False, paged=False,
             layers=1, V=1024, dtype="f32", sigma=1.0, p=0.7),
        # One layer's verification attention for a single user: LLaVA-v1.6-7B
        # (every query head has its own K/V, one image's tokens plus text).
        dict(name="attn_llava7b", kind=ATTN, B=1, T=60, depth=6, Hq=32, Hkv=32, D=128, L=3392, ragged=False,
             paged=False, lse=False),
        # The same for a grouped-query model: Qwen2-VL-7B, 7 query heads share
        # one K/V head; little memory traffic, short.
        dict(name="attn_qwen2vl7b", kind=ATTN, B=1, T=48, depth=5, Hq=28, Hkv=4, D=128, L=2000, ragged=False,
             paged=False, lse=False),
        # Batched serving: 16 users, ragged lengths and trees, paged cache.
        dict(name="attn_batched", kind=ATTN, B=16, T=64, depth=6, Hq=32, Hkv=8, D=128, L=6000, ragged=True, paged=True,
             lse=False),
        # A layer's prefill with the attention entropy that the choice of the
        # distillation layer averages.
        dict(name="prefill_llava7b", kind=MODES, mode="causal", B=1, T=3392, Hq=32, Hkv=32, D=128, L=0, ragged=False,
             paged=False, entropy=True),
        # The verification tail for a single user with the whole model's cache
        # (32 layers) compacted, f32 logits.
        dict(name="verify_llava7b", kind=VERIFY, B=1, T=60, depth=6, Hkv=32, D=128, L=3392, ragged=False, paged=False,
             layers=32, V=32000, dtype="f32", sigma=2.0, p=0.75),
        # The verification tail of batched serving, bf16 logits, large vocabulary.
        dict(name="verify_batched", kind=VERIFY, B=16, T=64, depth=6, Hkv=8, D=128, L=6000, ragged=True, paged=True,
             layers=1, V=128256, dtype="bf16", sigma=2.0, p=0.7),
        # The tail at temperature 1 for a few users; a vocabulary of 32000 plus
        # added special tokens, so rows do not start on 16 bytes.
        dict(name="sampled_oddvocab", kind=SAMPLED, B=4, T=60, depth=6, Hkv=32, D=128, L=3392, ragged=True, paged=True,
             layers=4, V=32003, dtype="f32", sigma=2.0, p=0.75, tau=1.0),
        # Speculative sampling over the tree in batched serving.
        dict(name="speculative_batched", kind=SPECULATIVE, B=16, T=64, depth=6, Hkv=8, D=128, L=6000, ragged=True,
             paged=True, layers=1, V=128256, dtype="bf16", sigma=2.0, p=0.7, tau=1.0),
        # The LM head for one user's tree: the weights are read once, few rows.
        dict(name="lm_head_qwen2vl7b", kind=LM_HEAD, rows=48, hidden=3584, V=152064),
        # The LM head of batched serving: compute-bound, the largest call.
        dict(name="lm_head_batched", kind=LM_HEAD, rows=854, hidden=4096, V=128256),
        # Visual-token selection from the last layer's prefill attention.
        dict(name="importance_llava7b", kind=IMPORTANCE, B=1, H=32, Q=3392, K=3392, v0=35, n_vis=2880, r=576,
             dtype="bf16"),
    ]


# ------------------------------------------------------------------ drawn cases
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _heads(rng):
    return rng.choice([(32, 32, 128), (28, 4, 128), (40, 40, 128), (32, 8, 128), (12, 2, 128), (16, 16, 64),
                       (4, 4, 64)])


def _tree(rng):
    T = rng.randint(1, 64)
    return T, max(1, min(T - 1, rng.randint(1, 8)))


def _vocab(rng):
    """(V, dtype): the vocabularies of common models, some with a few added tokens."""
    V = rng.choice([1024, 32000, 128256, 152064, _log(rng, 500, 160000)])
    if rng.random() < 0.25:
        V += rng.randint(1, 7)
    return V, rng.choice(["f32", "bf16"])


def _attention_ranges(rng):
    Hq, Hkv, D = _heads(rng)
    B = rng.choice([1, 1, _log(rng, 2, 16)])
    # one layer's K and V of the batch: at most 1 GB
    L = _log(rng, 16, max(17, min(16000, 2 ** 30 // (4 * Hkv * D * B))))
    return dict(B=B, Hq=Hq, Hkv=Hkv, D=D, L=L, ragged=B > 1 and rng.random() < 0.8, paged=rng.random() < 0.5)


def _tail_ranges(rng):
    c = _attention_ranges(rng)
    T, depth = _tree(rng)
    V, dtype = _vocab(rng)
    c["L"] = min(c["L"], 6000)
    most = max(1, 2 ** 31 // (4 * c["Hkv"] * c["D"] * c["B"] * (c["L"] + 64)))
    return dict(c, T=T, depth=depth, V=V, dtype=dtype, layers=min(most, _log(rng, 1, 40)), sigma=2.0,
                p=round(rng.uniform(0.5, 0.9), 3))


def draw(rng):
    kind = rng.choice([STEP, ATTN, ATTN, ATTN, MODES, MODES, VERIFY, VERIFY, SAMPLED, SPECULATIVE, LM_HEAD, IMPORTANCE])
    if kind == ATTN:
        T, depth = _tree(rng)
        return dict(_attention_ranges(rng), kind=kind, T=T, depth=depth, lse=rng.random() < 0.3)
    if kind == STEP:
        return dict(_tail_ranges(rng), kind=kind)
    if kind == MODES:
        Hq, Hkv, D = _heads(rng)
        mode = rng.choice(["full", "causal"])
        if mode == "full":  # the draft's positions against the target's features
            B, T, L = _log(rng, 1, 4), rng.randint(1, 128), _log(rng, 64, 6000)
        else:  # a prompt, or its last part after a cached prefix
            B, T, L = 1, _log(rng, 100, 3392), rng.choice([0, _log(rng, 16, 2000)])
        return dict(kind=kind, mode=mode, B=B, T=T, Hq=Hq, Hkv=Hkv, D=D, L=L, ragged=B > 1, paged=rng.random() < 0.3,
                    entropy=B == 1 and rng.random() < 0.5)
    if kind in (VERIFY, SAMPLED, SPECULATIVE):
        c = dict(_tail_ranges(rng), kind=kind)
        del c["Hq"]
        if kind != VERIFY:
            c["tau"] = rng.choice([1.0, round(rng.uniform(0.3, 1.5), 3)])
        return c
    if kind == LM_HEAD:
        hidden = rng.choice([1536, 2048, 3584, 4096, 5120])
        V = rng.choice([32000, 128256, 152064, _log(rng, 8000, 150000)])
        rows = _log(rng, 1, max(16, 854 * 4096 * 128256 // (hidden * V)) if rng.random() < 0.3 else 128)
        return dict(kind=kind, rows=min(rows, 854), hidden=hidden, V=V)
    K = _log(rng, 200, 3392)
    n_vis = max(16, int(K * rng.uniform(0.3, 0.9)))
    v0 = rng.randint(0, K - n_vis)
    return dict(kind=kind, B=1, H=rng.choice([16, 28, 32]), Q=rng.choice([K, max(1, K // 3)]), K=K, v0=v0, n_vis=n_vis,
                r=max(1, int(n_vis * rng.uniform(0.05, 0.6))), dtype=rng.choice(["bf16", "bf16", "f32"]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, shape, dtype=torch.bfloat16, std=1.0):
    """N(0, std) of any size, drawn in pieces so that no large f32 copy exists."""
    out = torch.empty(shape, dtype=dtype, device=DEV)
    flat = out.view(-1)
    step = 1 << 27
    for i in range(0, flat.numel(), step):
        n = min(step, flat.numel() - i)
        flat[i:i + n] = torch.randn(n, generator=g, device=DEV) * std
    return out


def _lengths(case, rng):
    """Tree (or query) lengths and prefix lengths of the sequences."""
    B, T, L = case["B"], case["T"], case["L"]
    tl, kl = np.full(B, T, np.int32), np.full(B, L, np.int32)
    if case["ragged"]:
        tl = rng.integers(max(1, T // 2), T + 1, B).astype(np.int32)
        kl = rng.integers(max(1, L // 4), L + 1, B).astype(np.int32)
        tl[0], kl[-1] = T, L
    return tl, kl


def _parents(case, tl, rng):
    """Draft trees numbered level by level, `depth` levels, each node's parent
    drawn from the level before."""
    B, T = case["B"], case["T"]
    par = np.full((B, T), -1, np.int32)
    for b in range(B):
        n = int(tl[b]) - 1
        depth = min(case["depth"], n)
        prev, nxt = [0], 1
        for lvl in range(depth):
            w = n // depth + (1 if lvl < n % depth else 0)
            cur = range(nxt, nxt + w)
            par[b, nxt:nxt + w] = rng.choice(prev, w)
            prev, nxt = list(cur), nxt + w
    return par


def _cache(case, g, rng, tl, kl, layers):
    """KV cache tensors (random, every slot filled) and the page table."""
    B, Hkv, D = case["B"], case["Hkv"], case["D"]
    cap = case["L"] + case["T"]
    table = None
    if case["paged"]:
        per = -(-cap // PAGE)
        need = [-(-int(tl[b] + kl[b]) // PAGE) for b in range(B)]
        pool = B * per  # a pool that would hold every sequence at its longest
        order = rng.permutation(pool).astype(np.int32)
        tab, at = np.full((B, per), -1, np.int32), 0
        for b in range(B):
            tab[b, :need[b]] = order[at:at + need[b]]
            at += need[b]
        table = torch.from_numpy(tab).to(DEV)
        shape = (pool, PAGE, Hkv, D)
    else:
        shape = (B, cap, Hkv, D)
    if layers is not None:
        shape = (layers,) + shape
    return dreams.KVCache(_randn(g, shape), _randn(g, shape), table)


def _logits(case, g, rng, par, tl, tok):
    """N(0, sigma) logits; a node with children gets, with probability p, one
    child's token as a clear maximum (the target agrees with the draft)."""
    B, T, V = case["B"], case["T"], case["V"]
    dt = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    x = _randn(g, (B, T, V), dt, case["sigma"])
    at = []
    for b in range(B):
        for i in range(int(tl[b])):
            kids = np.flatnonzero(par[b, :int(tl[b])] == i)
            if len(kids) and rng.random() < case["p"]:
                at.append((b, i, int(tok[b, rng.choice(kids)])))
    if at:
        b, i, v = (torch.tensor(c, device=DEV) for c in zip(*at))
        x[b, i, v] = 8.0 * case["sigma"]
    return x


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _ints(*shape):
    return torch.zeros(shape, dtype=torch.int32, device=DEV)


def prepare(case, seed):
    g, rng = _gen(seed), np.random.default_rng(int(seed))
    kind = case["kind"]
    s = dict(kind=kind, case=case, status=_ints(1))
    if kind == LM_HEAD:
        rows, K, V = case["rows"], case["hidden"], case["V"]
        w = _randn(g, (V, K), std=0.02)
        h = _randn(g, (rows, K))
        # the prediction stands out in most rows, as a trained head's does
        tgt = torch.randint(V, (rows,), generator=g, device=DEV)
        h += torch.where(torch.rand(rows, 1, generator=g, device=DEV) < 0.75, 10.0, 0.0).to(h.dtype) * w[tgt]
        s.update(h=h, w=w, out=_ints(rows), top=torch.zeros(rows, device=DEV))
        return s
    if kind == IMPORTANCE:
        B, H, Q, K = case["B"], case["H"], case["Q"], case["K"]
        a = torch.empty((B, H, Q, K), dtype=torch.float32 if case["dtype"] == "f32" else torch.bfloat16, device=DEV)
        for b in range(B):
            for h in range(H):
                # some key positions draw more attention than others
                bias = 1.5 * torch.randn(K, generator=g, device=DEV)
                a[b, h] = torch.softmax(torch.randn((Q, K), generator=g, device=DEV) + bias, -1).to(a.dtype)
        s.update(attn=a)
        return s
    tl, kl = _lengths(case, rng)
    s.update(tree_len=_dev(tl), kv_len=_dev(kl))
    s["kv"] = _cache(case, g, rng, tl, kl, case.get("layers"))
    if "Hq" in case:
        shape = (case["B"], case["T"], case["Hq"], case["D"])
        s.update(q=_randn(g, shape), out=torch.zeros(shape, dtype=torch.bfloat16, device=DEV),
                 scale=1.0 / math.sqrt(case["D"]))
    if kind == MODES:
        return s
    par = _parents(case, tl, rng)
    if kind == ATTN:
        s["tree"] = dreams.Tree(_dev(par), _ints(*par.shape), s["tree_len"], s["kv_len"])
        # (rows past a sequence's tree_len are not written: they stay zero)
        s["lse"] = torch.zeros(s["q"].shape[:3], device=DEV) if case["lse"] else None
        return s
    V, B, T = case["V"], case["B"], case["T"]
    tok = rng.integers(0, V, par.shape).astype(np.int32)
    s["logits"] = _logits(case, g, rng, par, tl, tok)
    s["max_path"] = case["depth"] + 1
    s["pred"] = _ints(B, T)
    s["outputs"] = (_ints(B), _ints(B, s["max_path"]), _ints(B, s["max_path"]), _ints(B))
    if kind == SAMPLED:
        s["u"] = torch.rand((B, T), generator=g, device=DEV)
    if kind == SPECULATIVE:
        # a draft close to the target; half of the children's tokens are the
        # draft's likeliest at their parent, the rest random
        s["draft"] = s["logits"] + _randn(g, s["logits"].shape, s["logits"].dtype, 0.5)
        top = s["draft"].argmax(-1).cpu().numpy()
        for b in range(B):
            for i in range(1, int(tl[b])):
                if rng.random() < 0.5:
                    tok[b, i] = top[b, par[b, i]]
        s["u"] = torch.rand((B, T), generator=g, device=DEV)
        s["u2"] = torch.rand((B, T), generator=g, device=DEV)
    s["tree"] = dreams.Tree(_dev(par), _dev(tok), s["tree_len"], s["kv_len"])
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    kind, case = s["kind"], s["case"]
    if kind == ATTN:
        out, lse = dreams.tree_verify_attn(s["q"], s["kv"], s["tree"], s["scale"], out=s["out"], lse=s["lse"],
                                           status=s["status"])
        return [out, lse]
    if kind == STEP:
        dreams.tree_verify_attn(s["q"], s["kv"], s["tree"], s["scale"], out=s["out"], status=s["status"])
        r = dreams.verify_step(s["logits"], s["tree"], s["kv"], s["max_path"], argmax_out=s["pred"],
                               outputs=s["outputs"], status=s["status"])
        return dict(r, pred=s["pred"], attn=s["out"], k=s["kv"].k, v=s["kv"].v)
    if kind == MODES:
        mode = dreams.ATTN_FULL if case["mode"] == "full" else dreams.ATTN_CAUSAL
        return list(dreams.attention(s["q"], s["kv"], s["tree_len"], s["kv_len"], s["scale"], mode, out=s["out"],
                                     want_entropy=case["entropy"], status=s["status"]))
    if kind == VERIFY:
        r = dreams.verify_step(s["logits"], s["tree"], s["kv"], s["max_path"], argmax_out=s["pred"],
                               outputs=s["outputs"], status=s["status"])
        return dict(r, pred=s["pred"], k=s["kv"].k, v=s["kv"].v)
    if kind == SAMPLED:
        r = dreams.verify_step_sampled(s["logits"], s["tree"], s["kv"], s["max_path"], case["tau"], s["u"],
                                       sample_out=s["pred"], outputs=s["outputs"], status=s["status"])
        return dict(r, pred=s["pred"], k=s["kv"].k, v=s["kv"].v)
    if kind == SPECULATIVE:
        r = dreams.verify_step_speculative(s["logits"], s["draft"], s["tree"], s["kv"], s["max_path"], case["tau"],
                                           s["u"], s["u2"], outputs=s["outputs"], status=s["status"])
        return dict(r, k=s["kv"].k, v=s["kv"].v)
    if kind == LM_HEAD:
        return list(dreams.lm_head_argmax(s["h"], s["w"], out=s["out"], out_max=s["top"], status=s["status"]))
    return list(dreams.visual_importance(s["attn"], case["v0"], case["n_vis"], case["r"]))


# ------------------------------------------------------------------ what a pass cannot do without
def _mean_lengths(case):
    """Expected tree nodes and prefix slots over the batch."""
    B, T, L = case["B"], case["T"], case["L"]
    if not case["ragged"]:
        return B * T, B * L
    return T + (B - 1) * (max(1, T // 2) + T) / 2, L + (B - 1) * (max(1, L // 4) + L) / 2


def work(case):
    kind = case["kind"]
    if kind == LM_HEAD:
        r, K, V = case["rows"], case["hidden"], case["V"]
        return {"bytes": 2 * K * (V + r) + 8 * r, "flops": 2 * r * K * V}
    if kind == IMPORTANCE:
        el = 4 if case["dtype"] == "f32" else 2
        n = case["B"] * case["H"] * case["Q"] * case["n_vis"]
        return {"bytes": el * n + 4 * case["B"] * (case["n_vis"] + case["r"]), "flops": n}
    nodes, slots = _mean_lengths(case)
    B, D, Hkv = case["B"], case["D"], case["Hkv"]
    nb = fl = 0.0
    if kind in (ATTN, STEP, MODES):
        Hq = case["Hq"]
        keys = slots if case.get("mode") == "full" else slots + nodes
        nb += 4 * keys * Hkv * D + 4 * nodes * Hq * D
        per = slots / B + (nodes / B / 2 if case.get("mode") == "causal" else 0)
        fl += 4 * nodes * Hq * D * per
        if case.get("lse"):
            nb += 4 * nodes * Hq
        if case.get("entropy"):
            nb += 4 * nodes * Hq
            fl += 2 * nodes * Hq * per
    if kind in (VERIFY, STEP, SAMPLED, SPECULATIVE):
        el = 4 if case["dtype"] == "f32" else 2
        moved = B * min(case["depth"], 3) * case["layers"] * 2 * 2 * 2 * Hkv * D
        # speculative sampling needs the rows of visited nodes only: about four
        # nodes, target and draft
        rows = 8 * B if kind == SPECULATIVE else nodes
        nb += rows * case["V"] * el + moved
        fl += rows * case["V"]
    return {"bytes": nb, "flops": fl}


def tolerance(case):
    kind = case["kind"]
    if kind in (ATTN, MODES, STEP):
        # bf16 probabilities and outputs, f32 sums
        return {"rel": 1e-2, "max": 0.06}
    if kind == IMPORTANCE:
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.01}  # f32 sums; near-ties at the cut
    if kind == LM_HEAD:
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.005}  # f32 sums; near-ties
    if kind == SAMPLED:
        return {"rel": 0.0, "differ": 0.01}  # draws decided by f32 sums
    return "exact"


# ------------------------------------------------------------------ 64-bit restatement
def _rows_of(s, layer, b, which):
    """K or V rows of sequence b (slots in order) of one layer."""
    kv = s["kv"]
    x = getattr(kv, which)
    if kv.n_layers > 1 or x.dim() == 5:
        x = x[layer]
    if kv.page_table is None:
        return x[b]
    pages = kv.page_table[b]
    return x[pages[pages >= 0].long()].reshape(-1, kv.Hkv, kv.D)


def _exact_attention(s):
    case = s["case"]
    B, T, Hq, D = s["q"].shape
    Hkv = case["Hkv"]
    G = Hq // Hkv
    out = torch.zeros((B, T, Hq, D), dtype=torch.float64, device=DEV)
    lse = torch.zeros((B, T, Hq), dtype=torch.float64, device=DEV)
    ent = torch.zeros((B, T, Hq), dtype=torch.float64, device=DEV)
    tl, kl = s["tree_len"].tolist(), s["kv_len"].tolist()
    par = s["tree"].parent.tolist() if "tree" in s else None
    for b in range(B):
        n, L = tl[b], kl[b]
        mode = case.get("mode", "tree")
        keys = L if mode == "full" else L + n
        ok = torch.zeros((n, keys), dtype=torch.bool, device=DEV)
        ok[:, :L] = True
        if mode == "causal":
            ok[:, L:] = torch.tril(torch.ones((n, n), dtype=torch.bool, device=DEV))
        elif mode == "tree":
            anc = np.zeros((n, n), bool)
            for i in range(n):
                if i:
                    anc[i] = anc[par[b][i]]
                anc[i, i] = True
            ok[:, L:] = torch.from_numpy(anc).to(DEV)
        k, v = (_rows_of(s, 0, b, w)[:keys] for w in ("k", "v"))
        for g in range(Hkv):
            kd, vd = k[:, g].double(), v[:, g].double()
            for h in range(g * G, (g + 1) * G):
                x = (s["q"][b, :n, h].double() @ kd.T) * s["scale"]
                x.masked_fill_(~ok, -math.inf)
                lz = torch.logsumexp(x, -1)
                a = torch.exp(x - lz[:, None])
                out[b, :n, h] = a @ vd
                lse[b, :n, h] = lz
                ent[b, :n, h] = -torch.where(ok, a * (x - lz[:, None]), 0.0).sum(-1)
    return out, lse, ent


def _walk(s, choose):
    """Acceptance given a function that returns a sequence's path and emitted
    tokens; then the compacted caches."""
    B, mp, kl = s["case"]["B"], s["max_path"], s["kv_len"].tolist()
    acc, path = np.zeros(B, np.int32), np.full((B, mp), -1, np.int32)
    toks, new = np.full((B, mp), -1, np.int32), np.zeros(B, np.int32)
    kv = s["kv"]
    k, v = kv.k.clone(), kv.v.clone()
    for b in range(B):
        p, t = choose(b)
        acc[b], new[b] = len(p), kl[b] + len(p)
        path[b, :len(p)], toks[b, :len(p)] = p, t
        src, dst = kl[b] + np.array(p), kl[b] + np.arange(len(p))
        for x in (k, v):
            y = x if x.dim() == 5 else x[None]
            if kv.page_table is None:
                y[:, b, dst] = y[:, b, src]
            else:
                tab = kv.page_table[b].cpu().numpy()
                y[:, tab[dst // PAGE], dst % PAGE] = y[:, tab[src // PAGE], src % PAGE]
    return dict(accept_len=acc, path=path, out_tokens=toks, new_kv_len=new, k=k, v=v)


def _exact_greedy(s, pred):
    """The longest root path whose drafts equal their parents' predictions
    (equal lengths: the smallest path), then the prediction at its end."""
    par, tok, tl = (getattr(s["tree"], n).tolist() for n in ("parent", "tokens", "tree_len"))

    def choose(b):
        paths = {0: [0]}
        for i in range(1, tl[b]):
            up = par[b][i]
            if up in paths and tok[b][i] == pred[b][up]:
                paths[i] = paths[up] + [i]
        best = min(paths.values(), key=lambda p: (-len(p), p))[:s["max_path"]]
        return best, [tok[b][i] for i in best[1:]] + [pred[b][best[-1]]]

    return _walk(s, choose)


def _draw(w, u):
    """The first entry where the running sum of weights exceeds u times their sum."""
    c = torch.cumsum(w, -1)
    return int(torch.searchsorted(c, u * c[-1], right=True).clamp(max=w.numel() - 1))


def _exact_speculative(s):
    par, tok, tl = (getattr(s["tree"], n).tolist() for n in ("parent", "tokens", "tree_len"))
    tau, ua, ur = s["case"]["tau"], s["u"].double(), s["u2"].double()

    def choose(b):
        path, emitted = [0], []
        while True:
            cur = path[-1]
            r = torch.softmax(s["logits"][b, cur].double() / tau, -1)
            q = torch.softmax(s["draft"][b, cur].double() / tau, -1)
            nxt = None
            kids = [i for i in range(1, tl[b]) if par[b][i] == cur] if len(path) < s["max_path"] else []
            for c in kids:
                x = tok[b][c]
                if float(ua[b, c]) < (min(1.0, float(r[x] / q[x])) if float(q[x]) > 0 else float(r[x] > 0)):
                    nxt = c
                    break
                left = torch.clamp(r - q, min=0)
                if float(left.sum()) > 0:
                    r = left / left.sum()
            if nxt is None:
                return path, emitted + [_draw(r, ur[b, cur])]
            path.append(nxt)
            emitted.append(tok[b][nxt])

    return _walk(s, choose)


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == ATTN:
        out, lse, _ = _exact_attention(s)
        return [out, lse if case["lse"] else None]
    if kind == MODES:
        out, _, ent = _exact_attention(s)
        return [out, None, ent if case["entropy"] else None]
    if kind == LM_HEAD:
        best = torch.full((case["rows"],), -math.inf, dtype=torch.float64, device=DEV)
        idx = torch.zeros(case["rows"], dtype=torch.int64, device=DEV)
        h = s["h"].double()
        for v0 in range(0, case["V"], 16384):
            x, i = (h @ s["w"][v0:v0 + 16384].double().T).max(-1)
            idx = torch.where(x > best, i + v0, idx)
            best = torch.maximum(x, best)
        return [idx.int(), best]
    if kind == IMPORTANCE:
        v0, n = case["v0"], case["n_vis"]
        imp = torch.zeros((case["B"], n), dtype=torch.float64, device=DEV)
        for h in range(case["H"]):
            imp += s["attn"][:, h, :, v0:v0 + n].sum(1, dtype=torch.float64)
        imp /= case["H"] * case["Q"]
        keep = torch.sort(imp, dim=-1, descending=True, stable=True).indices[:, :case["r"]].sort(-1).values + v0
        return [imp, keep.int()]
    if kind == SPECULATIVE:
        return _exact_speculative(s)
    if kind == SAMPLED:
        pred = _ints(case["B"], case["T"])
        for b, n in enumerate(s["tree_len"].tolist()):
            for i in range(n):
                w = torch.exp((s["logits"][b, i].double() - s["logits"][b, i].double().max()) / case["tau"])
                pred[b, i] = _draw(w, s["u"][b, i].double())
    else:
        pred = s["logits"].double().argmax(-1).int()
        for b, n in enumerate(s["tree_len"].tolist()):
            pred[b, n:] = 0
    r = dict(_exact_greedy(s, pred.tolist()), pred=pred)
    if kind == STEP:
        r["attn"] = _exact_attention(s)[0]
    return r
