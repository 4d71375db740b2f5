"""GPU parity at the sizes where the attention's segments and merges and the LM
head's CTA pairs and top-K lists can go wrong: CTAs that walk more segments than
the published ring holds, row blocks of a few rows split over many CTAs, a row of
NaN scores, node counts around one node tile and the pair rule, odd numbers of
vocabulary tiles, list quarters with fewer rows than k.  References and tolerances are those
of the other parity tests (the fp64 oracle; parity_util)."""
import numpy as np
import pytest
import torch

import oracle as O
import parity_util as U
import test_gpu_verify as V
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    import paper_2506_02780_gb300 as E
    from paper_2506_02780_gb300 import build
    build.build_lib()
    E.lib()


@pytest.mark.parametrize("kind", ["tree", "inplace", "chain"])
@pytest.mark.parametrize("n_q,n_kv", [(8, 8), (24, 8)])
def test_many_short_segments(kind, n_q, n_kv):
    """400 sequences of 0 to 120 cached positions and 1 to 5 nodes: a balanced
    launch whose CTAs each walk about 20 segments of one or two tiles (more than
    the 16 the ring of published segments holds)."""
    import paper_2506_02780_gb300 as E
    from paper_2506_02780_gb300 import step as S
    rng = np.random.default_rng(7)
    B = 400
    Ts = rng.integers(1, 6, B)
    w = W.build("tiny", seed=71, device="cuda", vocab=512, hidden=64, n_q=n_q, n_kv=n_kv,
                trees=[W.TreeSpec(int(t), [], [0]) for t in Ts], ctxs=[int(c) for c in rng.integers(0, 121, B)])
    mode = {"tree": False, "inplace": True, "chain": "chain"}[kind]
    plan = E.ee_attn_plan(w.B, w.max_T, n_q, n_kv, int(w.ctx_len.max()), inplace=mode)
    assert plan["mode"] == "balanced"
    kc, vc = (torch.from_numpy(U.raw16(t).copy()).view(torch.bfloat16) for t in (w.k_cache, w.v_cache))
    st = S.from_workload(w, inplace_kv=kind == "inplace", chain=kind == "chain")
    st.run()
    torch.cuda.synchronize()
    assert E.ee_read_errors(st.ws) == 0
    anc = O.tree_prepare(w.parent, w.node_off)[1]
    ref = O.tree_attention(w.q[0], w.k_tree[0], w.v_tree[0], kc[0], vc[0], w.block_table, w.ctx_len, w.node_off, anc)
    U.assert_close(st.attn_out[0].cpu().numpy(), ref, f"{kind} attention")


@pytest.mark.parametrize("T,ctx", [(1, 3001), (2, 129), (3, 1999), (19, 2500), (64, 4096)])
def test_few_rows_split_over_many_ctas(T, ctx):
    """One sequence, 28 / 4 heads: row blocks of 7 to 128 rows cut into up to 15
    chunks, merged by column chunks."""
    import paper_2506_02780_gb300 as E
    from paper_2506_02780_gb300 import step as S
    w = W.build("7b", seed=72, device="cuda", layers=1, vocab=512, hidden=64, trees=[W.TreeSpec(T, [], [0])], ctx=ctx)
    kc, vc = (torch.from_numpy(U.raw16(t).copy()).view(torch.bfloat16) for t in (w.k_cache, w.v_cache))
    st = S.from_workload(w)
    st.run()
    torch.cuda.synchronize()
    assert E.ee_read_errors(st.ws) == 0
    anc = O.tree_prepare(w.parent, w.node_off)[1]
    ref = O.tree_attention(w.q[0], w.k_tree[0], w.v_tree[0], kc[0], vc[0], w.block_table, w.ctx_len, w.node_off, anc)
    U.assert_close(st.attn_out[0].cpu().numpy(), ref, f"T = {T}, ctx = {ctx}")


@pytest.mark.parametrize("B,ctx,T,n_q,n_kv,kind", [(16, 60, 60, 28, 4, "tree"), (16, 60, 120, 28, 4, "inplace"),
                                                   (1, 72, 560, 56, 8, "chain"), (4, 300, 133, 56, 8, "chain")])
def test_uniform_plans_beside_the_balanced_line(B, ctx, T, n_q, n_kv, kind):
    """Two or three waves of whole row blocks, close to where the plan changes to
    the balanced launch: ragged contexts and draft sizes below the plan's maxima."""
    import paper_2506_02780_gb300 as E
    import test_gpu_chain
    import test_gpu_inplace
    from paper_2506_02780_gb300 import step as S
    rng = np.random.default_rng(9)
    ctxs = [ctx] + [int(c) for c in rng.integers(0, ctx + 1, B - 1)]
    Ts = [T] + [int(t) for t in rng.integers(1, T + 1, B - 1)]
    w = W.build("long" if kind == "chain" else "tiny", seed=76, device="cuda", layers=1, vocab=512, hidden=64,
                n_q=n_q, n_kv=n_kv, trees=[W.TreeSpec(t, [], [0]) for t in Ts], ctxs=ctxs)
    mode = {"tree": False, "inplace": True, "chain": "chain"}[kind]
    assert E.ee_attn_plan(w.B, w.max_T, n_q, n_kv, ctx, inplace=mode)["mode"] != "balanced"
    if kind == "chain":
        test_gpu_chain.check_chain_attention(w, nodes=sorted(set(rng.integers(0, w.total_nodes, 128).tolist())))
    elif kind == "inplace":
        test_gpu_inplace.check_inplace(w, layers=[0])
    else:
        kc, vc = (torch.from_numpy(U.raw16(t).copy()).view(torch.bfloat16) for t in (w.k_cache, w.v_cache))
        st = S.from_workload(w)
        st.run()
        torch.cuda.synchronize()
        assert E.ee_read_errors(st.ws) == 0
        anc = O.tree_prepare(w.parent, w.node_off)[1]
        ref = O.tree_attention(w.q[0], w.k_tree[0], w.v_tree[0], kc[0], vc[0], w.block_table, w.ctx_len, w.node_off,
                               anc)
        U.assert_close(st.attn_out[0].cpu().numpy(), ref, "tree attention")


@pytest.mark.parametrize("seed,first,last", [(81, 3.505e-6, 3.685e-6), (82, 3.329e-6, 3.504e-6),
                                             (83, 3.398e-6, 3.573e-6)])
def test_long_sums_add_the_tails_first(seed, first, last):
    """1,500 keys in one CTA, whose accumulator each P.V MMA cuts at its lowest bits: the
    relative error (2-norm) against fp64 with a tile's tails added before its heads
    (`first`), not the 5 % larger one of the other order (`last`).  Seeded inputs, sums in
    a fixed order: the bound is half way between the two."""
    import paper_2506_02780_gb300 as E
    from paper_2506_02780_gb300 import step as S
    w = W.build("tiny", seed=seed, device="cuda", vocab=512, hidden=64, trees=[W.TreeSpec(64, [], [0])], ctxs=[1500])
    kc, vc = (torch.from_numpy(U.raw16(t).copy()).view(torch.bfloat16) for t in (w.k_cache, w.v_cache))
    st = S.from_workload(w)
    st.ws = E.new_workspace(1, 64, 1, 0)      # no partial slots: one CTA per row block
    st.run()
    torch.cuda.synchronize()
    assert E.ee_read_errors(st.ws) == 0
    anc = O.tree_prepare(w.parent, w.node_off)[1]
    ref = O.tree_attention(w.q[0], w.k_tree[0], w.v_tree[0], kc[0], vc[0], w.block_table, w.ctx_len, w.node_off, anc)
    err = np.linalg.norm(st.attn_out[0].cpu().numpy() - ref) / np.linalg.norm(ref)
    assert err < (first + last) / 2


@pytest.mark.parametrize("ctxs", [[512], [2900] * 40])
def test_nan_scores_stay_in_their_row(ctxs):
    """A query row of NaN (split and balanced launches): its output is NaN, every
    other row is bit-identical to a run without it, and no wait gives up."""
    import paper_2506_02780_gb300 as E
    from paper_2506_02780_gb300 import step as S
    w = W.build("tiny", seed=73, device="cuda", vocab=512, hidden=64,
                trees=[W.TreeSpec(12, [(0, 4)], [0]) for _ in ctxs], ctxs=ctxs)
    st = S.from_workload(w)
    st.run()
    torch.cuda.synchronize()
    clean = st.attn_out[0].clone()
    w.q[0, 3, 2] = float("nan")
    st.run()
    torch.cuda.synchronize()
    assert E.ee_read_errors(st.ws) == 0
    got = st.attn_out[0]
    assert torch.isnan(got[3, 2]).all()
    keep = torch.ones(got.shape[:2], dtype=torch.bool, device=got.device)
    keep[3, 2] = False
    assert torch.equal(got[keep], clean[keep])


def test_query_offsets_beyond_four_gib():
    """A causal draft of 2,048 nodes with 8,320 query heads: the byte offset of a
    node's query rows passes 2^32 from node 2,017 on.  Sampled rows on both sides
    against fp64."""
    import paper_2506_02780_gb300 as E
    T, n_q, n_kv = 2048, 8320, 65
    gen = torch.Generator(device="cuda").manual_seed(77)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    q = torch.empty((T, n_q, 128), **bf).normal_(generator=gen)
    assert 2016 * n_q * 256 < 2**32 <= 2017 * n_q * 256
    kc, vc = (torch.empty((T // 16, n_kv, 16, 128), **bf).normal_(generator=gen) for _ in range(2))
    i32 = dict(dtype=torch.int32, device="cuda")
    bt = torch.arange(T // 16, **i32).view(1, -1)
    out = torch.full((T, n_q, 128), float("nan"), device="cuda")
    ws = E.new_workspace(1, T, 1, 0)      # no partial slots: one CTA per row block
    E.ee_chain_verify_attn(q, kc, vc, bt, torch.zeros(1, **i32), 0, torch.tensor([0, T], **i32), T, 128**-0.5, out, ws)
    torch.cuda.synchronize()
    assert E.ee_read_errors(ws) == 0
    for node in (0, 1000, 2016, 2017, 2047):
        for head in (0, 4099, n_q - 1):
            k, v = (c[:, head * n_kv // n_q].reshape(T, 128)[:node + 1].double() for c in (kc, vc))
            ref = torch.softmax(k @ q[node, head].double() * 128**-0.5, 0) @ v
            U.assert_close(out[node, head].cpu().numpy(), ref.cpu().numpy(), f"node {node} head {head}")


@pytest.mark.parametrize("nodes,vocab,hidden,packed", [(256, 4100, 512, True), (513, 4097, 520, False),
                                                       (1025, 4100, 64, False), (96, 4100, 3584, True),
                                                       (97, 4100, 3592, False), (192, 4097, 2048, True),
                                                       (193, 4097, 2048, True), (256, 8320, 3584, False),
                                                       (257, 4100, 2056, False), (513, 4224, 2048, True)])
def test_lmhead_around_the_pair_line(nodes, vocab, hidden, packed):
    """Node counts and hidden sizes on both sides of the lines between CTAs of
    their own and CTA pairs, one node tile (up to 256 nodes) and several, with odd
    numbers of 128-row vocabulary tiles: argmax, longest prefix and logits."""
    import paper_2506_02780_gb300 as E
    w = W.build("long", seed=74, device="cuda", layers=1, vocab=vocab, hidden=hidden, n_q=8, n_kv=2,
                trees=[W.TreeSpec(nodes, [], W.chain_path(nodes // 2))], ctxs=[16])
    i32 = dict(dtype=torch.int32, device="cuda")
    ws = E.new_workspace(1, nodes, 1, 0)
    am, acc, bonus = (torch.empty(n, **i32) for n in (nodes, 1, 1))
    path = torch.empty((1, nodes), **i32)
    logits = torch.full((nodes, vocab), float("nan"), device="cuda")
    node_off = torch.as_tensor(w.node_off, **i32)
    draft = torch.as_tensor(w.draft_tok, **i32)
    for _ in range(2):   # the running state returns to zero after a call
        if packed:
            wp = torch.empty(E.ee_lmhead_packed_bytes(vocab, hidden) // 2, dtype=torch.bfloat16, device="cuda")
            E.ee_lmhead_pack_weights(w.lm_w, wp)
            E.ee_lmhead_accept_packed(w.hidden_states, wp, vocab, draft, None, None, None, node_off, nodes, am, acc,
                                      path, bonus, ws, logits=logits)
        else:
            E.ee_lmhead_accept(w.hidden_states, w.lm_w, draft, None, None, None, node_off, nodes, am, acc, path,
                               bonus, ws, logits=logits)
        torch.cuda.synchronize()
        assert E.ee_read_errors(ws) == 0
    U.check_argmax(w, type("S", (), {"argmax": am})(), logits=logits)
    ra, rp, rb = O.accept_chain(am.cpu().numpy(), w.draft_tok, w.node_off, nodes)
    np.testing.assert_array_equal(acc.cpu().numpy(), ra)
    np.testing.assert_array_equal(path.cpu().numpy(), rp)
    np.testing.assert_array_equal(bonus.cpu().numpy(), rb)


@pytest.mark.parametrize("mode,k,hidden,trees", [("entropy", 5, 3584, 6), ("entropy", 5, 2048, 15),
                                                 ("topk", 8, 2048, 15), ("topk", 8, 512, 15)])
def test_verify_with_many_nodes(mode, k, hidden, trees):
    """6 or 15 trees of 20 nodes: the verification rules on CTA pairs with one and
    with two node tiles, and on CTAs of their own with two."""
    w = W.build("tiny", seed=75, device="cuda", hidden=hidden, verify_plant=True, trees=[V.TREE] * trees)
    V._check(w, V._run(w, mode, k), mode, k)


@pytest.mark.parametrize("vocab", [40, 130, 200, 29792])
@pytest.mark.parametrize("k", [2, 8])
def test_verify_lists_with_few_rows(vocab, k):
    """Lists that a tile fills only in part (a quarter of 32 rows holds 0, 2 or 8
    of them; at 29,792 words 2 of a first tile's 98 rows, and a second tile inserts):
    top-k ids, entropy and acceptance."""
    w = W.build("tiny", seed=76, device="cuda", vocab=vocab)
    V._check(w, V._run(w, "entropy", k), "entropy", k)


@pytest.mark.parametrize("vocab", [4096, 4100, 29792])
@pytest.mark.parametrize("mode,k", [("topk", 1), ("topk", 8), ("entropy", 5)])
def test_verify_with_nan_words(vocab, mode, k):
    """Vocabulary rows of NaN -- beside node 0's best word, in every quarter of a
    tile, nine in a row (more than a list holds); at 4,100 words the last tile's only
    four -- and a node whose logits are all NaN (one and two tiles a CTA): no NaN word
    is chosen or ranked, the other words rank as without them, H_norm is 0 and top_tau 1."""
    w = W.build("tiny", seed=78, device="cuda", verify_plant=True, trees=[V.TREE], vocab=vocab)
    lg, err = O.lm_head_logits(w.hidden_states, w.lm_w)
    best = O.node_ranking(lg[0], 3).tolist()
    words = {best[0] ^ 1, 3, 40, 70, 100, 161} | set(range(600, 609)) if vocab % 128 != 4 else set(range(4096, 4100))
    words = sorted(words - set(best))
    w.lm_w[words] = float("nan")
    w.hidden_states[5] = float("nan")
    r = V._run(w, mode, k)
    assert r["argmax"][5] == -1 and (r["topk"][5] == 2**31 - 1).all()
    lg[:, words] = -np.inf
    for a in range(w.total_nodes):
        if a == 5:
            continue
        ids = r["topk"][a]
        assert r["argmax"][a] == ids[0] and len(set(ids.tolist())) == k and not set(ids.tolist()) & set(words), a
        e = 2.0 * err[a].max()      # fp32 accumulation: closer words may change places
        np.testing.assert_allclose(lg[a][ids], lg[a][O.node_ranking(lg[a], k)], atol=e, rtol=0)
    if mode == "entropy":
        assert (r["h"] == 0).all() and (r["tau"] == 1).all()
    g = V._run(w, "greedy", 1, verify=False)
    np.testing.assert_array_equal(g["argmax"], r["argmax"])
