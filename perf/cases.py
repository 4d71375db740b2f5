"""Performance cases of the verification step: what a program that uses libee has it do.

A server of edit sessions draws a draft tree for each sequence (reuse-span
match, tree build, tree preparation), runs one target pass over all trees
(tree-masked paged attention, every layer), decodes greedily or by the
entropy-aware rule (LM head + acceptance) and appends the accepted K/V to the
cache.  The cases are these calls at the sizes of the configurations (tiny,
7B-shaped, batched ragged, 33B-shaped, long reuse draft, match / compaction
sweep) and, by ``draw``, over the ranges between and around them.

Values: K and V are N(0, 1/128) as in the synthetic workloads, queries
N(0, 16^2), which gives scores of standard deviation 1.4 (a peaked but not
degenerate softmax); LM-head weights N(0, 0.02^2); a node's hidden state is 12
times the unit vector of its target's weight row plus N(0, 1) noise, so that the
greedy choice has the margin of a trained model and no near ties.

Lengths come from the case alone (``sizes`` seeds them), values from the seed.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2506_02780_gb300 as E
from paper_2506_02780_gb300.step import VerifyStep

D = 128
PAGE = 16
DEV = "cuda"

# attention heads / LM head of the target models the configurations are shaped after
TINY = dict(n_q=8, n_kv=2, hidden=512, vocab=4096)
M7 = dict(n_q=28, n_kv=4, hidden=3584, vocab=152064)
M33 = dict(n_q=56, n_kv=8, hidden=7168, vocab=32256)


def _attn(shape, **k):
    return dict(dict(kind="attn", inplace=False, layers=1, graph=False, n_q=shape["n_q"], n_kv=shape["n_kv"]), **k)


def _lm(shape, **k):
    return dict(dict(kind="lmhead", chain=False, packed=False, logits=False, hidden=shape["hidden"],
                     vocab=shape["vocab"]), **k)


def listed():
    return [
        # the smallest whole step: every kernel is a few microseconds, launches and latency are all
        dict(TINY, name="step-tiny", kind="step", B=1, ctx_lo=512, ctx_hi=512, t_lo=16, t_hi=16, layers=1,
             code=400, n=4, sizes=1),
        # one step of an edit session on a 7B-shaped target: 28 layers, 64-node tree, captured as a server does
        dict(M7, name="step-7b", kind="step", B=1, ctx_lo=4096, ctx_hi=4096, t_lo=64, t_hi=64, layers=28, code=3000,
             n=4, sizes=1),
        # no match and no draft: the pass scores the root alone (plain decoding), four layers captured
        _attn(M7, name="attn-root-only", B=1, ctx_lo=3001, ctx_hi=3001, t_lo=1, t_hi=1, layers=4, graph=True, sizes=1),
        # long file, 128-node tree, 33B-shaped: one layer
        _attn(M33, name="attn-33b", B=1, ctx_lo=32768, ctx_hi=32768, t_lo=128, t_hi=128, sizes=1),
        # eight edit sessions of ragged lengths in one pass
        _attn(M7, name="attn-batched", B=8, ctx_lo=1024, ctx_hi=16384, t_lo=32, t_hi=96, sizes=7),
        # in-place speculative K/V: a few sessions of ordinary length, odd sizes
        _attn(M7, name="attn-inplace", B=4, ctx_lo=777, ctx_hi=8191, t_lo=17, t_hi=63, inplace=True, layers=4,
              graph=True, sizes=3),
        # a 2048-token reuse draft verified in one pass (causal): prefill-like
        dict(kind="chain", name="chain-long", n_q=28, n_kv=4, B=1, ctx_lo=4096, ctx_hi=4096, t_lo=2048, t_hi=2048,
             sizes=1),
        # greedy LM head on the checkpoint's own (row-major) weights, logits kept for a sampler
        _lm(M33, name="lmhead-33b-logits", B=1, t_lo=128, t_hi=128, logits=True, sizes=1),
        # greedy LM head of the batched step on tile-ordered weights
        _lm(M7, name="lmhead-batched", B=8, t_lo=32, t_hi=96, packed=True, sizes=7),
        # entropy-aware verification, the paper's larger setting k = 5
        dict(M7, kind="verify", name="verify-entropy", B=1, t_lo=64, t_hi=64, mode="entropy", k=5, sizes=1),
        # draft construction for 32 sessions with 64k-token codes: match, tree build, tree preparation, captured
        dict(kind="draft", name="draft-sweep", B=32, code_lo=65536, code_hi=65536, n=4, vocab=152064, chain_len=48,
             branches=2, gen_len=8, sizes=1),
        # accepted paths of 32 sessions appended to the cache, 28 layers
        dict(kind="compact", name="compact-sweep", B=32, n_kv=4, layers=28, t_lo=128, t_hi=128, a_lo=1, a_hi=128,
             ctx_lo=0, ctx_hi=1024, sizes=1),
    ]


def _logi(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attn", "attn", "attn", "chain", "lmhead", "lmhead", "verify", "draft", "compact", "step"])
    shape = rng.choice([TINY, M7, M33])
    sizes = rng.randrange(1, 1 << 20)
    if kind == "attn":
        B = _logi(rng, 1, 16)
        # no more keys times query rows than the long-file case: 32768 x 128 x 56
        hi = _logi(rng, 64, max(64, min(32768, 32768 * 56 // (B * shape["n_q"]))))
        lo = rng.randrange(0, hi + 1)
        t_hi = _logi(rng, 1, 128)
        return _attn(shape, B=B, ctx_lo=lo, ctx_hi=hi, t_lo=rng.randrange(1, t_hi + 1), t_hi=t_hi,
                     inplace=rng.random() < 0.4, sizes=sizes)
    if kind == "chain":
        B = rng.choice([1, 1, 2, 4])
        t = _logi(rng, 129, 2048 // B)
        hi = _logi(rng, 64, 16384 // B)
        return dict(kind="chain", n_q=shape["n_q"], n_kv=shape["n_kv"], B=B, ctx_lo=rng.randrange(0, hi + 1),
                    ctx_hi=hi, t_lo=rng.randrange(129, t + 1), t_hi=t, sizes=sizes)
    if kind == "lmhead":
        chain = rng.random() < 0.25
        B = 1 if chain else _logi(rng, 1, 8)
        t = _logi(rng, 1, 640) if chain else _logi(rng, 1, 96)
        return _lm(shape, B=B, t_lo=t if chain else rng.randrange(1, t + 1), t_hi=t, chain=chain,
                   packed=rng.random() < 0.5, logits=rng.random() < 0.2, sizes=sizes)
    if kind == "verify":
        t = _logi(rng, 1, 96)
        return dict(shape, kind="verify", B=rng.choice([1, 1, 2, 3]), t_lo=rng.randrange(1, t + 1), t_hi=t,
                    mode=rng.choice(["entropy", "entropy", "topk"]), k=rng.choice([2, 3, 3, 5, 5, 8]), sizes=sizes)
    if kind == "draft":
        hi = _logi(rng, 256, 65536)
        chain = rng.randrange(1, 49)
        return dict(kind="draft", B=_logi(rng, 1, 32), code_lo=rng.randrange(256, hi + 1), code_hi=hi,
                    n=rng.choice([1, 2, 4, 8, 11]), vocab=shape["vocab"], chain_len=chain, branches=rng.randrange(1, 3),
                    gen_len=rng.randrange(0, 9), sizes=sizes)
    if kind == "compact":
        t = _logi(rng, 1, 128)
        hi = rng.randrange(0, 4096)
        return dict(kind="compact", B=_logi(rng, 1, 32), n_kv=shape["n_kv"], layers=rng.randrange(1, 29), t_lo=t,
                    t_hi=t, a_lo=1, a_hi=t, ctx_lo=rng.randrange(0, hi + 1), ctx_hi=hi, sizes=sizes)
    hi = _logi(rng, 64, 4096)
    t = _logi(rng, 1, 64)
    return dict(rng.choice([TINY, M7]), kind="step", B=1, ctx_lo=rng.randrange(0, hi + 1), ctx_hi=hi, t_lo=t, t_hi=t,
                layers=rng.randrange(1, 9), code=_logi(rng, 256, 8000), n=rng.choice([2, 4, 8]), sizes=sizes)


# ---------------------------------------------------------------- sizes (from the case alone)

def _lengths(case):
    """Per sequence (context length, tree nodes)."""
    r = random.Random(case["sizes"])
    B = case["B"]
    ctx = [r.randint(case.get("ctx_lo", 0), case.get("ctx_hi", 0)) for _ in range(B)]
    T = [r.randint(case["t_lo"], case["t_hi"]) for _ in range(B)]
    if B > 1:
        ctx[-1], T[0] = case.get("ctx_hi", 0), case["t_hi"]
    return ctx, T


def _parents(T, r):
    """A reuse chain (root first, 50 to 90 % of the nodes) and two generated branches below it."""
    chain = max(1, min(T, int(round(T * r.uniform(0.5, 0.9)))))
    rest = T - chain
    par = [-1] + list(range(chain - 1))
    for attach, length in ((0, rest // 2), (r.randrange(chain), rest - rest // 2)):
        for j in range(length):
            par.append(attach if j == 0 else len(par) - 1)
    return par, chain


def _trees(case):
    """Local parent ids of every sequence's tree, the chain lengths, and the nodes' depths."""
    _, Ts = _lengths(case)
    r = random.Random(case["sizes"] + 1)
    parents, chains, depths = [], [], []
    for T in Ts:
        par, chain = (list(range(-1, T - 1)), T) if case.get("chain") or case["kind"] == "chain" else _parents(T, r)
        dep = []
        for p in par:
            dep.append(0 if p < 0 else dep[p] + 1)
        parents.append(par)
        chains.append(chain)
        depths.append(dep)
    return parents, chains, depths


def _codes(case):
    r = random.Random(case["sizes"] + 2)
    return [r.randint(case["code_lo"], case["code_hi"]) for _ in range(case["B"])]


def _accepts(case):
    r = random.Random(case["sizes"] + 3)
    return [r.randint(case["a_lo"], min(case["a_hi"], t)) - 1 for t in _lengths(case)[1]]


# ---------------------------------------------------------------- inputs

def _randn(gen, shape, std):
    out = torch.empty(shape, dtype=torch.bfloat16, device=DEV)
    flat = out.view(-1)
    for a in range(0, flat.numel(), 1 << 27):
        n = min(1 << 27, flat.numel() - a)
        flat[a:a + n] = torch.randn(n, generator=gen, device=DEV) * std
    return out


def _gens(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    return gen, np.random.Generator(np.random.PCG64(int(seed)))


def _i32(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.int32).to(DEV)


def _pages(nrng, ctx, T, extra=3):
    """Block table (pages of each sequence in random order) for ctx + T positions per sequence, as wide as
    the longest context and the largest tree together need."""
    per = [max(1, -(-(c + t) // PAGE)) for c, t in zip(ctx, T)]
    num = sum(per) + extra
    perm = nrng.permutation(num)
    bt = np.full((len(per), -(-(max(ctx) + max(T)) // PAGE)), -1, dtype=np.int32)
    o = 0
    for s, p in enumerate(per):
        bt[s, :p] = perm[o:o + p]
        o += p
    return bt, num


def _kv_inputs(case, seed):
    gen, nrng = _gens(seed)
    ctx, T = _lengths(case)
    L, n_q, n_kv = case.get("layers", 1), case["n_q"], case["n_kv"]
    bt, num = _pages(nrng, ctx, T)
    total = sum(T)
    std = D ** -0.5
    x = dict(q=_randn(gen, (L, total, n_q, D), 16.0), k_cache=_randn(gen, (L, num, n_kv, PAGE, D), std),
             v_cache=_randn(gen, (L, num, n_kv, PAGE, D), std))
    if not case.get("inplace") and case["kind"] != "chain":
        x["k_tree"] = _randn(gen, (L, total, n_kv, D), std)
        x["v_tree"] = _randn(gen, (L, total, n_kv, D), std)
    x.update(block_table=_i32(bt), ctx_len=_i32(ctx), node_off=_i32(np.concatenate([[0], np.cumsum(T)])))
    x["parent"] = _i32(np.concatenate([np.asarray(p) for p in _trees(case)[0]]))
    return x, max(ctx), max(T), total


def _lm_inputs(case, seed, second=False):
    """Weights, hidden states and drafts whose planted path is accepted to a random depth.  With
    `second`, a node's second choice comes close to its first (edit content is uncertain)."""
    gen, nrng = _gens(seed + 17)
    parents, chains, _ = _trees(case)
    V, H = case["vocab"], case["hidden"]
    W = _randn(gen, (V, H), 0.02)
    tok, tgt = [], []
    for par, chain in zip(parents, chains):
        T = len(par)
        t = nrng.integers(0, V, T)
        g = nrng.integers(0, V, T)
        for a in range(int(nrng.integers(0, chain))):   # the reuse chain is accepted this far
            g[a] = t[a + 1]
        tok.append(t)
        tgt.append(g)
    tgt = torch.as_tensor(np.concatenate(tgt)).to(DEV)
    unit = torch.nn.functional.normalize(W[tgt].float(), dim=1)
    h = torch.randn((len(tgt), H), generator=gen, device=DEV) + 12.0 * unit
    if second:
        alt = torch.as_tensor(nrng.integers(0, V, len(tgt))).to(DEV)
        w = torch.as_tensor(nrng.uniform(6.0, 12.0, len(tgt)), dtype=torch.float32).to(DEV)
        h += w[:, None] * torch.nn.functional.normalize(W[alt].float(), dim=1)
    gen_mask = np.concatenate([np.arange(len(p)) >= c for p, c in zip(parents, chains)]).astype(np.uint8)
    return W, h.to(torch.bfloat16), _i32(np.concatenate(tok)), torch.as_tensor(gen_mask).to(DEV)


def _code_inputs(case, seed, lens, V, n):
    """Codes with repeated segments and tails copied from them: ambiguous matches."""
    _, nrng = _gens(seed + 29)
    codes, tails, cursors = [], [], []
    for m in lens:
        c = nrng.integers(0, V, m)
        for _ in range(max(1, m // 64)):
            a, b = nrng.integers(0, m - 8, 2)
            c[b:b + 8] = c[a:a + 8].copy()
        cur = int(nrng.integers(0, m // 2))
        p = int(nrng.integers(cur, m - n))
        codes.append(c)
        tails.append(c[p:p + n] if nrng.random() < 0.9 else nrng.integers(0, V, n))
        cursors.append(cur)
    off = np.concatenate([[0], np.cumsum(lens)])
    return dict(orig_tokens=_i32(np.concatenate(codes)), orig_off=torch.as_tensor(off, dtype=torch.int64).to(DEV),
                tail=_i32(np.stack(tails)), cursor=_i32(cursors))


def _captured(fn):
    """The calls of fn as a CUDA graph, as a server keeps its step."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        fn()
        s.synchronize()
        with torch.cuda.graph(g, stream=s):
            fn()
    torch.cuda.current_stream().wait_stream(s)
    return g


def _new_i32(*shape):
    return torch.zeros(shape, dtype=torch.int32, device=DEV)


# ---------------------------------------------------------------- prepare / run

def prepare(case, seed):
    st = dict(globals()["_prepare_" + case["kind"]](case, seed), case=case)
    if case["kind"] in ("step", "draft") or case.get("graph"):
        st["graph"] = _captured(lambda: st["go"]())
    return st


def run(state):
    if "graph" in state:
        state["graph"].replay()
    else:
        state["go"]()
    return state["out"]


def _prepare_attn(case, seed):
    x, max_ctx, max_T, total = _kv_inputs(case, seed)
    L, B = case["layers"], case["B"]
    out = torch.zeros((L, total, case["n_q"], D), dtype=torch.float32, device=DEV)
    ws = E.new_workspace(B, total, case["n_q"], max_ctx)
    depth, anc = _new_i32(total), torch.zeros((total, 2), dtype=torch.int64, device=DEV)
    E.ee_tree_prepare(x["parent"], x["node_off"], depth, anc, ws)
    scale = D ** -0.5

    def go():
        for l in range(L):
            if case["inplace"]:
                E.ee_tree_verify_attn_inplace(x["q"][l], x["k_cache"][l], x["v_cache"][l], x["block_table"],
                                              x["ctx_len"], max_ctx, x["node_off"], anc, max_T, scale, out[l], ws)
            else:
                E.ee_tree_verify_attn(x["q"][l], x["k_tree"][l], x["v_tree"][l], x["k_cache"][l], x["v_cache"][l],
                                      x["block_table"], x["ctx_len"], max_ctx, x["node_off"], anc, max_T, scale,
                                      out[l], ws)
    return dict(go=go, out=out, x=x)


def _prepare_chain(case, seed):
    x, max_ctx, max_T, total = _kv_inputs(case, seed)
    out = torch.zeros((1, total, case["n_q"], D), dtype=torch.float32, device=DEV)
    ws = E.new_workspace(case["B"], total, case["n_q"], max_ctx)

    def go():
        E.ee_chain_verify_attn(x["q"][0], x["k_cache"][0], x["v_cache"][0], x["block_table"], x["ctx_len"], max_ctx,
                               x["node_off"], max_T, D ** -0.5, out[0], ws)
    return dict(go=go, out=out, x=x)


def _lm_outputs(case, total, max_T):
    return dict(argmax=_new_i32(total), accept_len=_new_i32(case["B"]), path=_new_i32(case["B"], max_T),
                bonus=_new_i32(case["B"]))


def _tree_arrays(case, ws):
    parents, _, _ = _trees(case)
    node_off = _i32(np.concatenate([[0], np.cumsum([len(p) for p in parents])]))
    parent = _i32(np.concatenate([np.asarray(p) for p in parents]))
    depth = _new_i32(parent.numel())
    anc = torch.zeros((parent.numel(), 2), dtype=torch.int64, device=DEV)
    if not case.get("chain"):
        E.ee_tree_prepare(parent, node_off, depth, anc, ws)
    return node_off, parent, depth, anc


def _prepare_lmhead(case, seed):
    W, h, tok, _ = _lm_inputs(case, seed)
    total, V = h.shape[0], case["vocab"]
    ws = E.new_workspace(case["B"], total, 1, 0)
    node_off, parent, depth, anc = _tree_arrays(case, ws)
    if case["chain"]:
        parent = depth = anc = None
    max_T = max(_lengths(case)[1])
    out = _lm_outputs(case, total, max_T)
    if case["logits"]:
        out["logits"] = torch.zeros((total, V), dtype=torch.float32, device=DEV)
    if case["packed"]:
        Wp = torch.empty(E.ee_lmhead_packed_bytes(V, case["hidden"]) // 2, dtype=torch.bfloat16, device=DEV)
        E.ee_lmhead_pack_weights(W, Wp)
        W = Wp

    def go():
        a = (tok, parent, depth, anc, node_off, max_T, out["argmax"], out["accept_len"], out["path"], out["bonus"], ws)
        if case["packed"]:
            E.ee_lmhead_accept_packed(h, W, V, *a, logits=out.get("logits"))
        else:
            E.ee_lmhead_accept(h, W, *a, logits=out.get("logits"))
    return dict(go=go, out=out)


def _prepare_verify(case, seed):
    W, h, tok, mask = _lm_inputs(case, seed, second=True)
    total = h.shape[0]
    ws = E.new_workspace(case["B"], total, 1, 0)
    node_off, parent, depth, anc = _tree_arrays(case, ws)
    max_T = max(_lengths(case)[1])
    out = _lm_outputs(case, total, max_T)
    out.update(topk_ids=_new_i32(total, case["k"]), top_tau=_new_i32(total),
               h_norm=torch.zeros(total, dtype=torch.float32, device=DEV))

    def go():
        E.ee_lmhead_verify(h, W, tok, parent, depth, anc, node_off, max_T, case["mode"], case["k"], out["argmax"],
                           out["accept_len"], out["path"], out["bonus"], ws, gen_mask=mask, topk_ids=out["topk_ids"],
                           top_tau=out["top_tau"], h_norm=out["h_norm"])
    return dict(go=go, out=out)


def _prepare_draft(case, seed):
    B, n = case["B"], case["n"]
    lens = _codes(case)
    x = _code_inputs(case, seed, lens, case["vocab"], n)
    _, nrng = _gens(seed + 31)
    T = 1 + case["branches"] * case["chain_len"] + case["gen_len"]
    last = x["tail"][:, -1].contiguous()
    gen_tok = _i32(nrng.integers(0, case["vocab"], (B, case["gen_len"]))) if case["gen_len"] else None
    ws = E.new_workspace(B, B * T, 1, 0)
    out = dict(match_pos=_new_i32(B, 8), n_matches=_new_i32(B), draft_tok=_new_i32(B * T), parent=_new_i32(B * T),
               node_off=_new_i32(B + 1), cpos=_new_i32(B * T),
               gen_mask=torch.zeros(B * T, dtype=torch.uint8, device=DEV), depth=_new_i32(B * T),
               anc=torch.zeros((B * T, 2), dtype=torch.int64, device=DEV))

    def go():
        E.ee_match_reuse(x["orig_tokens"], x["orig_off"], x["tail"], x["cursor"], 8, out["match_pos"],
                         out["n_matches"], ws)
        E.ee_build_reuse_tree(x["orig_tokens"], x["orig_off"], out["match_pos"], out["n_matches"], last, n,
                              case["chain_len"], case["branches"], out["draft_tok"], out["parent"], out["node_off"],
                              out["cpos"], out["gen_mask"], ws, gen_tok=gen_tok)
        E.ee_tree_prepare(out["parent"], out["node_off"], out["depth"], out["anc"], ws)
    return dict(go=go, out=out)


def _prepare_compact(case, seed):
    gen, nrng = _gens(seed)
    ctx, T = _lengths(case)
    acc = _accepts(case)
    B, L, n_kv, max_T, total = case["B"], case["layers"], case["n_kv"], max(T), sum(T)
    bt, num = _pages(nrng, ctx, T)
    kt, vt = (_randn(gen, (L, total, n_kv, D), D ** -0.5) for _ in range(2))
    kc, vc = (_randn(gen, (L, num, n_kv, PAGE, D), D ** -0.5) for _ in range(2))
    path = np.full((B, max_T), -1, dtype=np.int32)
    for s, a in enumerate(acc):   # an accepted path through a tree: ascending node ids, the root first
        path[s, 1:a + 1] = np.sort(nrng.choice(np.arange(1, T[s]), a, replace=False))
        path[s, 0] = 0
    path, acc, bt = _i32(path), _i32(acc), _i32(bt)
    node_off, ctx_in = _i32(np.concatenate([[0], np.cumsum(T)])), _i32(ctx)
    ws = E.new_workspace(B, total, 1, 0)
    out = dict(k_cache=kc, v_cache=vc, ctx_out=_new_i32(B), dst_slot=_new_i32(B, max_T))

    def go():
        E.ee_kv_compact(kt, vt, kc, vc, bt, ctx_in, out["ctx_out"], node_off, path, acc, out["dst_slot"], ws)
    return dict(go=go, out=out)


def _prepare_step(case, seed):
    x, max_ctx, max_T, total = _kv_inputs(case, seed)
    W, h, tok, _ = _lm_inputs(case, seed)
    code = _code_inputs(case, seed, [case["code"]] * case["B"], case["vocab"], case["n"])
    vs = VerifyStep(**code, parent=x["parent"], node_off=x["node_off"], draft_tok=tok, ctx_len=x["ctx_len"],
                    block_table=x["block_table"], q=x["q"], k_tree=x["k_tree"], v_tree=x["v_tree"],
                    k_cache=x["k_cache"], v_cache=x["v_cache"], hidden=h, lm_w=W, max_ctx=max_ctx, max_T=max_T)
    logits = torch.zeros((total, case["vocab"]), dtype=torch.float32, device=DEV)
    for t in (vs.outputs, vs.dst_slot, vs.attn_out):
        t.zero_()
    out = dict(attn=vs.attn_out, logits=logits, match_pos=vs.match_pos, n_matches=vs.n_matches, argmax=vs.argmax,
               accept_len=vs.accept_len, path=vs.path, bonus=vs.bonus, ctx_out=vs.ctx_out, dst_slot=vs.dst_slot,
               k_cache=x["k_cache"], v_cache=x["v_cache"])
    return dict(go=lambda: vs.run(logits=logits), out=out, vs=vs)


# ---------------------------------------------------------------- work, tolerance, exact

def _attn_work(case):
    ctx, T = _lengths(case)
    _, _, depths = _trees(case)
    n_q, n_kv = case["n_q"], case["n_kv"]
    by = sum(2 * (c + t) * n_kv * D * 2 + t * n_q * D * (2 + 4) for c, t in zip(ctx, T))
    fl = sum(4 * n_q * D * sum(c + d + 1 for d in dep) for c, dep in zip(ctx, depths))
    return case.get("layers", 1) * by, case.get("layers", 1) * fl


def _lm_work(case, logits):
    total = sum(_lengths(case)[1])
    V, H = case["vocab"], case["hidden"]
    return V * H * 2 + total * H * 2 + total * 4 * 4 + (total * V * 4 if logits else 0), 2 * total * V * H


def work(case):
    kind = case["kind"]
    if kind in ("attn", "chain"):
        by, fl = _attn_work(case)
    elif kind == "lmhead":
        by, fl = _lm_work(case, case["logits"])
    elif kind == "verify":
        by, fl = _lm_work(case, False)
    elif kind == "draft":
        T = 1 + case["branches"] * case["chain_len"] + case["gen_len"]
        by, fl = sum(3 * m for m in _codes(case)) + case["B"] * T * (3 * 4 + 1 + 4 + 16), 0   # cursor at a quarter
    elif kind == "compact":
        by, fl = 2 * 2 * sum(a + 1 for a in _accepts(case)) * case["layers"] * case["n_kv"] * D * 2, 0
    else:
        b1, f1 = _attn_work(case)
        b2, f2 = _lm_work(case, True)
        by, fl = b1 + b2, f1 + f2
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """About four times the measured distance from 64 bits at the worst listed case of the kind."""
    kind = case["kind"]
    if kind in ("draft", "compact"):
        return "exact"
    if kind in ("attn", "chain"):
        # fp32 softmax and sums, P carried as two bf16 parts: 2.6e-5 over 32k keys, 1e-5 over 16k, 2e-6 over 3k
        return {"rel": 1e-4, "max": 1e-3}
    if kind == "lmhead":
        # fp32 sums of 7168 bf16 products: 7.9e-6
        return {"rel": 3e-5, "max": 3e-4, "differ": 0.002}
    if kind == "verify":
        # fp32 log-sum-exp over the vocabulary: h_norm 1e-5; a rank may change hands between near ties
        return {"rel": 4e-5, "max": 1e-3, "differ": 0.004}
    # a step: attention over at most 4k keys 2.7e-6, logits 3.8e-6
    return {"rel": 2e-5, "max": 4e-4, "differ": 0.002}


def _exact_attn(x, case, ctx, T, parents):
    """softmax(q k / sqrt(d)) v in 64 bits, node by visible keys, every layer and KV head."""
    L, n_q, n_kv = case.get("layers", 1), case["n_q"], case["n_kv"]
    g = n_q // n_kv
    out = torch.zeros((L, sum(T), n_q, D), dtype=torch.float64, device=DEV)
    o = 0
    for s, (c, t) in enumerate(zip(ctx, T)):
        vis = torch.zeros((t, t), dtype=torch.bool, device="cpu")
        for i, p in enumerate(parents[s]):
            if p >= 0:
                vis[i] = vis[p]
            vis[i, i] = True
        vis = torch.cat([torch.ones((t, c), dtype=torch.bool), vis], dim=1).to(DEV)
        pos = torch.arange(c + t, device=DEV)
        page = x["block_table"][s].long()[pos // PAGE]
        for l in range(L):
            for kv in range(n_kv):
                k, v = (x[n][l][page, kv, pos % PAGE].double() for n in ("k_cache", "v_cache"))
                if "k_tree" in x:
                    k[c:], v[c:] = (x[n][l, o:o + t, kv].double() for n in ("k_tree", "v_tree"))
                q = x["q"][l, o:o + t, kv * g:(kv + 1) * g].double()
                for h in range(g):
                    p = (q[:, h] @ k.T) * D ** -0.5
                    p.masked_fill_(~vis, -math.inf)
                    out[l, o:o + t, kv * g + h] = torch.softmax(p, dim=1) @ v
        o += t
    return out


def _exact_logits(W, h):
    out = torch.empty((h.shape[0], W.shape[0]), dtype=torch.float64, device=DEV)
    hd = h.double()
    for a in range(0, W.shape[0], 16384):
        out[:, a:a + 16384] = hd @ W[a:a + 16384].double().T
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("draft", "compact") or (kind == "lmhead" and not case["logits"]):
        return None
    none = dict.fromkeys(("argmax", "accept_len", "path", "bonus"))
    if kind in ("attn", "chain"):
        return _exact_attn(_kv_inputs(case, seed)[0], case, *_lengths(case), _trees(case)[0])
    if kind == "lmhead":
        W, h, _, _ = _lm_inputs(case, seed)
        return dict(none, logits=_exact_logits(W, h))
    if kind == "verify":
        W, h, _, _ = _lm_inputs(case, seed, second=True)
        lg = _exact_logits(W, h)
        lp = torch.topk(lg, case["k"], dim=1).values - torch.logsumexp(lg, dim=1, keepdim=True)
        return dict(none, topk_ids=None, top_tau=None, h_norm=-(lp.exp() * lp).sum(1) / math.log(case["k"]))
    x = _kv_inputs(case, seed)[0]
    W, h, _, _ = _lm_inputs(case, seed)
    return dict(none, attn=_exact_attn(x, case, *_lengths(case), _trees(case)[0]), logits=_exact_logits(W, h),
                **dict.fromkeys(("match_pos", "n_matches", "ctx_out", "dst_slot", "k_cache", "v_cache")))
