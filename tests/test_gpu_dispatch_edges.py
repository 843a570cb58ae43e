"""The kernels that a dispatch chooses by size, at the edges of their ranges, against the oracle: products of few and
many tokens (through prefilling and its K/V rows), the draft heads' top-k, and the sampled root with ties at the edge
of the nucleus."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle import sampling as S
from harness import TOL, read_kv, tokens_with_phonemes

pytestmark = pytest.mark.gpu


def _prefill_rows_match(dtype, chunks, last, check, nodes=64, d_ffn=1024):
    """`chunks` sequences of one chunk each (the last of `last` tokens) in one pass; K/V rows of the checked ones."""
    import paper_2410_21951_b200 as P
    wl = W.toy_workload(dtype=dtype, d_model=256, n_heads=4, d_ffn=d_ffn, vocab=203, tree_nodes=16, tree_caps=(6, 3, 2),
                        batch=chunks, index=31)
    w = W.make_weights(wl.shape, wl.seed())
    model = O.Model.from_shape(wl.shape, w)
    lens = [nodes] * (chunks - 1) + [last]
    ph = [W.phonemes(min(9, n), wl.shape.n_phonemes, wl.seed(b)) for b, n in enumerate(lens)]
    pr = [W.markov_prompt(n - len(ph[b]), wl.shape.vocab - 1, wl.seed(b)) for b, n in enumerate(lens)]
    mat = np.zeros((chunks, nodes), dtype=np.int32)
    for b, n in enumerate(lens):
        mat[b, :n] = tokens_with_phonemes(wl.shape, ph[b], pr[b])
    table, total = W.shuffled_block_table(lens, 64, 5, spare_pages=2)
    g = P.Vadusa(wl.shape, w, max_batch=chunks, max_tree_nodes=nodes, max_blocks_per_seq=table.shape[1], kv_num_blocks=total)
    g.begin(table)
    g.prefill(mat, lens)
    assert list(g.lengths()) == lens
    for b in check:
        st = O.prefill_blocked(model, ph[b], pr[b], seq=b)
        K, V = read_kv(g, table, b, lens[b])
        assert np.abs(K - st.kv.K[:, :lens[b]]).max() <= TOL[dtype], b
        assert np.abs(V - st.kv.V[:, :lens[b]]).max() <= TOL[dtype], b
    g.check()
    g.close()


# 256 and 1024 features: every tile width of the pair products, with the last token tile full or not
@pytest.mark.parametrize("chunks,last", [(2, 64), (3, 1), (5, 37), (17, 64), (33, 5), (65, 64), (98, 33), (114, 64), (130, 9)])
def test_bf16_products_of_many_tokens(chunks, last):
    _prefill_rows_match("bf16", chunks, last, sorted({0, chunks // 2, chunks - 1}))


# up to 64 tokens the K slices of a product are merged by the tokens of a tile: 2, 4, 8 and 16 slices, tiles full or not
@pytest.mark.parametrize("tokens,d_ffn", [(2, 1024), (15, 512), (16, 1024), (17, 512), (31, 1024), (33, 512), (63, 1024), (64, 512)])
def test_bf16_split_products_of_few_tokens(tokens, d_ffn):
    _prefill_rows_match("bf16", 1, tokens, [0], nodes=tokens, d_ffn=d_ffn)


# the few-token product kernel serves up to 128 rows of a pass, the tile kernel beyond
@pytest.mark.parametrize("chunks,last,nodes", [(1, 1, 16), (1, 3, 4), (1, 5, 5), (2, 7, 64), (2, 64, 64), (3, 1, 43), (3, 2, 64)])
def test_fp32_products_around_the_few_token_limit(chunks, last, nodes):
    _prefill_rows_match("fp32", chunks, last, range(chunks), nodes=nodes)


@pytest.mark.parametrize("vocab,topk", [(2, 1), (17, 16), (255, 10), (257, 10), (4096, 16), (4097, 10), (12000, 16)])
@pytest.mark.parametrize("tied", [False, True])
def test_draft_topk_at_vocabulary_edges(vocab, topk, tied):
    """Identity draft block and one-hot hidden state: the logits are a column of the vocabulary matrix."""
    import torch
    import paper_2410_21951_b200 as P
    d, heads, batch = 16, 2, 3
    rng = np.random.default_rng(vocab + topk)
    u = np.zeros((heads, (vocab + 127) // 128 * 128, d), dtype=np.float32)
    vals = rng.standard_normal((heads, vocab, batch)).astype(np.float32)
    if tied:
        vals = np.round(vals)                                             # a handful of values: ties everywhere
    u[:, :vocab, :batch] = vals
    h = np.zeros((batch, d), dtype=np.float32)
    h[np.arange(batch), np.arange(batch)] = 1.0
    dev = torch.device("cuda")
    t = lambda a: torch.from_numpy(a).to(dev)
    out = torch.full((batch, heads, topk), -7, dtype=torch.int32, device=dev)
    P.draft_topk_static(t(np.zeros((heads, d, d), np.float32)), t(np.zeros((heads, d), np.float32)), t(u), t(h), 0, batch, d,
                        vocab, heads, topk, False, out)
    got = out.cpu().numpy()
    for b in range(batch):
        for i in range(heads):
            want = np.lexsort((np.arange(vocab), -vals[i, :, b]))[:topk]   # larger logit, then lower id
            assert list(got[b, i]) == list(want), (b, i)


@pytest.mark.parametrize("vocab", [5, 300, 4096, 4100])
@pytest.mark.parametrize("top_p", [0.05, 0.5, 0.9, 0.999])
@pytest.mark.parametrize("levels", [0, 1, 4])
def test_root_sample_with_ties_at_the_edge_of_the_nucleus(vocab, top_p, levels):
    """levels = 0: distinct logits; else that many values, so that the nucleus ends inside a run of equal ones."""
    import torch
    import paper_2410_21951_b200 as P
    wl = W.toy_workload(dtype="fp32", vocab=vocab, n_draft_heads=1, tree_nodes=2, tree_caps=(1,), batch=6, index=33)
    sh = wl.shape
    table, total = W.shuffled_block_table([70] * 6, 64, 3)
    g = P.Vadusa(sh, W.make_weights(sh, 1), max_batch=6, max_tree_nodes=2, max_blocks_per_seq=table.shape[1], kv_num_blocks=total,
                 draft_topk=1)
    g.begin(table)
    tpl = W.chain_template(2)
    g.set_tree(tpl.parent, tpl.rank)
    rng = np.random.default_rng(vocab)
    lg = rng.standard_normal((6, vocab)).astype(np.float32) * 2
    if levels:
        lg = rng.integers(0, levels, size=(6, vocab)).astype(np.float32)
    g.load_state(torch.zeros(6, sh.d_model, device=g.dev), torch.from_numpy(lg).to(g.dev))
    tokens = torch.zeros(6, 2, dtype=torch.int32, device=g.dev)
    compared = 0
    for seed in range(4):
        g.draft(P.Sampling.make(tau=1, temperature=1.0, top_p=top_p, seed=seed), tree_tokens=tokens)
        got = tokens.cpu().numpy()[:, 0]
        for b in range(6):
            l32 = S.masked_logits32(lg[b], sh.eos_id, True)
            keys = S.decision_keys(l32, 1.0, seed, b, 0)
            # fp32 sums may put the boundary a token to either side: compare where that does not decide
            roots = {S.root_token(keys, S.nucleus_sorted(l32, 1.0, min(top_p + e, 0.99999))) for e in (-1e-5, 0.0, 1e-5)}
            nucleus = S.nucleus_sorted(l32, 1.0, top_p)
            two = np.sort(np.where(nucleus, keys, -np.inf))[::-1][:2]
            if len(roots) == 1 and two[0] - two[1] > 1e-4:
                assert got[b] in roots, (b, seed)
                compared += 1
    assert compared > 0
    g.close()
