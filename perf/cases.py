"""Performance cases of the tree draft-and-verify library: what a program that serves a speech-token model asks of it.

A server keeps one context per model (weights, paged KV pool, workspace) and many requests; here the contexts are kept
per process (`_context`), a case's state owns pages of the pool, and `run` is one request or one burst of iterations.

The weights are random with the repository's standard deviation, except that token embeddings dominate the residual
stream and the vocabulary heads carry a successor table (token t is followed by succ(t); draft head i knows the token
i + 2 places on for most t): the base model's distribution is peaked and the draft heads are right most of the time, as
in a trained model, so that a pass commits about three tokens and the sampled tokens do not hang on rounding.
"""
from __future__ import annotations

import weakref
from dataclasses import replace

import numpy as np
import torch

import paper_2410_21951_b200 as P
import workloads as W

CAPS = (10, 5, 3, 2)                 # usable top-k ranks per draft depth
HEAD_HIT = (0.85, 0.75, 0.65, 0.55)  # share of tokens for which draft head i proposes the right token first
MEAN_ACCEPTED = 3.1                  # tokens per iteration that these heads give
SLOTS = 5                            # requests (states) whose pages a context's pool can hold at once

_VALLE = W.workload("C2").shape
MODELS = {
    # shape, context: tokens of pool pages per request, largest batch, tree nodes, prefill chunks per pass, blocks per sequence
    "tiny_fp32": (W.workload("C1").shape, dict(tokens=16384, batch=8, nodes=64, rows=16, blocks=64)),
    "valle_1025": (_VALLE, dict(tokens=131072, batch=64, nodes=64, rows=256, blocks=80)),
    "valle_1025_n128": (_VALLE, dict(tokens=32768, batch=16, nodes=128, rows=16, blocks=80)),
    "valle_2049": (W.workload("C3").shape, dict(tokens=32768, batch=32, nodes=42, rows=64, blocks=64)),
    "small_16001": (replace(_VALLE, n_layers=2, d_model=256, n_heads=4, d_ffn=1024, vocab=16001),
                    dict(tokens=16384, batch=8, nodes=64, rows=16, blocks=64)),
}


def listed():
    return [
        # offline synthesis with the smallest model, fp32, greedy: every launch is short, latency counts
        dict(name="generate_fp32_tiny", kind="generate", model="tiny_fp32", batch=1, nodes=16, prefix_lo=107, prefix_hi=107,
             new_tokens=100, tau=1, temperature=0.0, top_p=1.0),
        # one utterance of ten seconds: prefix in host memory to tokens in host memory
        dict(name="generate_b1", kind="generate", model="valle_1025", batch=1, nodes=64, prefix_lo=325, prefix_hi=325,
             new_tokens=750, tau=3, temperature=1.0, top_p=1.0),
        # a batch of utterances, 50 Hz tokens of a larger vocabulary, nucleus sampling
        dict(name="generate_b16_nucleus", kind="generate", model="valle_2049", batch=16, nodes=42, prefix_lo=190, prefix_hi=270,
             new_tokens=500, tau=5, temperature=0.8, top_p=0.9),
        # a streaming server that calls draft, verify and accept itself: one long utterance
        dict(name="steps_b1_ctx2600", kind="steps", model="valle_1025", batch=1, nodes=64, ctx_lo=2600, ctx_hi=2600, iterations=4,
             tau=3, temperature=1.0, top_p=1.0),
        # the same with a handful of utterances in flight
        dict(name="steps_b8", kind="steps", model="valle_1025", batch=8, nodes=64, ctx_lo=300, ctx_hi=1200, iterations=4,
             tau=3, temperature=1.0, top_p=1.0),
        # long-context serving, ragged contexts
        dict(name="steps_b32_long", kind="steps", model="valle_1025", batch=32, nodes=64, ctx_lo=1000, ctx_hi=4000, iterations=4,
             tau=3, temperature=1.0, top_p=1.0),
        # the largest vocabulary (a 16000-entry codebook) on a small model, nucleus sampling
        dict(name="steps_b2_vocab16001", kind="steps", model="small_16001", batch=2, nodes=48, ctx_lo=150, ctx_hi=400, iterations=4,
             tau=4, temperature=0.9, top_p=0.95),
        # a tree of its own per sequence, candidates from the caller, scores returned
        dict(name="verify_b64", kind="verify", model="valle_1025", batch=64, nodes=64, ctx_lo=256, ctx_hi=3000,
             tau=3, temperature=1.0, top_p=1.0),
        # the larger candidate trees
        dict(name="verify_b2_nodes128", kind="verify", model="valle_1025_n128", batch=2, nodes=128, ctx_lo=325, ctx_hi=1100,
             tau=3, temperature=1.0, top_p=1.0),
        # prefilling: one short prefix (time to the first token), and a batch of long ragged ones
        dict(name="prefill_b1", kind="prefill", model="valle_1025", batch=1, prefix_lo=325, prefix_hi=325),
        dict(name="prefill_b32_long", kind="prefill", model="valle_1025", batch=32, prefix_lo=1000, prefix_hi=4000),
        # fitting the draft heads with the base model frozen: two optimiser steps (forward, backward, update)
        dict(name="fit_512", kind="fit", model="valle_1025", dtype="bf16", tokens=512, steps=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["generate", "steps", "steps", "verify", "verify", "prefill", "fit"])
    if kind == "fit":
        return dict(kind=kind, model="valle_1025", dtype=rng.choice(["bf16", "bf16", "fp32"]), tokens=_log_int(rng, 24, 700), steps=2)
    tau, temperature, top_p = rng.randint(1, 5), rng.choice([0.0, 0.8, 1.0]), rng.choice([1.0, 1.0, 0.9])
    if kind == "generate":
        model = rng.choice(["tiny_fp32", "valle_1025", "valle_2049"])
        lo = _log_int(rng, 40, 500)
        batch = _log_int(rng, 1, {"tiny_fp32": 8, "valle_1025": 16, "valle_2049": 16}[model])
        return dict(kind=kind, model=model, batch=batch, nodes=rng.randint(10, 42), prefix_lo=lo, prefix_hi=lo + rng.randint(0, 150),
                    new_tokens=_log_int(rng, 20, 400), tau=1 if batch > 1 else tau, temperature=temperature, top_p=top_p)
    if kind == "prefill":
        lo = _log_int(rng, 30, 2000)
        return dict(kind=kind, model="valle_1025", batch=_log_int(rng, 1, 24), prefix_lo=lo, prefix_hi=lo + _log_int(rng, 10, 1900))
    lo = _log_int(rng, 64, 2000)
    ctx = dict(ctx_lo=lo, ctx_hi=lo + _log_int(rng, 10, 1500))
    if kind == "verify":
        model = rng.choice(["valle_1025", "valle_1025", "valle_1025_n128"])
        nodes = rng.randint(8, 64) if model == "valle_1025" else rng.randint(65, 128)
        return dict(kind=kind, model=model, batch=_log_int(rng, 1, 40 if model == "valle_1025" else 8), nodes=nodes, **ctx,
                    tau=tau, temperature=temperature, top_p=top_p)
    model = rng.choice(["valle_1025", "valle_1025", "small_16001"])
    return dict(kind=kind, model=model, batch=_log_int(rng, 1, 32 if model == "valle_1025" else 4), nodes=rng.randint(8, 64), **ctx,
                iterations=4, tau=tau, temperature=temperature, top_p=top_p)


# ---- the model and its context ---------------------------------------------------------------------------------------

def _zeros_for(shape, cfg):
    """Placeholder weights of the right shapes; `_fill_weights` writes the real ones on the GPU."""
    return {t.name.decode(): np.broadcast_to(np.float32(0), (t.rows, t.cols) if t.is_matrix else (t.rows,))
            for t in P.tensor_infos(cfg)}


def _fill_weights(g, seed):
    """The model's weights, drawn on the GPU into the blob.  Returns what a case needs of them: the direction of every
    token's embedding, the base head's matrix and the successor table."""
    sh, gen = g.shape, torch.Generator(device=g.dev).manual_seed(seed)
    info = {t.name.decode(): t for t in P.tensor_infos(g.cfg)}

    def normal(rows, cols, std, mean=0.0):
        return torch.randn(rows, cols, generator=gen, device=g.dev) * std + mean

    def put(name, value):
        t = info[name]
        raw = g.blob[t.offset:t.offset + t.nbytes]
        if t.is_matrix:
            raw.view(g.tdtype).view(t.rows_padded, t.cols)[:t.rows] = value.to(g.tdtype)
        else:
            raw.view(torch.float32)[:] = value.reshape(-1)

    for name, t in info.items():
        gain = name.endswith(("ln1_g", "ln2_g", "lnf_g"))
        std = {"emb_audio": 2.0, "emb_phon": 2.0, "pos": 0.1}.get(name, 0.02)
        put(name, normal(t.rows, t.cols, std, 1.0 if gain else 0.0))
    n = sh.vocab - 1                                                       # the last id is EOS
    unit = torch.randn(n, sh.d_model, generator=gen, device=g.dev)
    emb = info["emb_audio"]
    g.blob[emb.offset:emb.offset + emb.nbytes].view(g.tdtype).view(emb.rows, emb.cols)[:n] = (2.0 * unit).to(g.tdtype)
    order = torch.randperm(n, generator=gen, device=g.dev)
    succ = torch.empty_like(order)
    succ[order] = torch.roll(order, -1)                                    # one cycle through all ids
    row_std = 24.0 / sh.d_model
    heads = [("lm", succ, 1.0)]
    step = succ
    for i in range(sh.n_draft_heads):
        step = succ[step]
        heads.append((f"draft{i}.u", step, HEAD_HIT[min(i, 3)]))
    lm = None
    for name, target, hit in heads:
        wrong = torch.nonzero(torch.rand(n, generator=gen, device=g.dev) >= hit).flatten()
        target = target.clone()
        target[wrong] = target[torch.roll(wrong, 1)]                       # these tokens' answers are swapped around
        m = normal(sh.vocab, sh.d_model, row_std)
        m[target] = row_std * unit
        put(name, m)
        lm = m.to(g.tdtype).float() if name == "lm" else lm
    return dict(unit=unit, lm=lm, succ=succ)


class _Context:
    """One model's context, its weights, and which pages of its pool belong to which request."""

    def __init__(self, model):
        self.shape, c = MODELS[model]
        self.pages_per_slot = c["tokens"] // 64
        cfg = P.Config.from_buffer_copy(_config(self.shape, c, SLOTS * self.pages_per_slot))
        self.g = P.Vadusa(self.shape, _zeros_for(self.shape, cfg), max_batch=c["batch"], max_tree_nodes=c["nodes"],
                          max_blocks_per_seq=c["blocks"], kv_num_blocks=SLOTS * self.pages_per_slot, prefill_rows=c["rows"])
        self.weights = _fill_weights(self.g, 1000)
        self.free = list(range(SLOTS))
        self.tree = None

    def set_tree(self, nodes):
        if self.tree != nodes:
            t = W.static_template(nodes, CAPS[:self.shape.n_draft_heads])
            self.g.set_tree(t.parent, t.rank)
            self.tree = nodes

    def pages(self, state, tokens, seed):
        """Block table over shuffled pages of a free slot: tokens[b] positions for sequence b."""
        table, n = W.shuffled_block_table(tokens, 64, seed)
        if not self.free or n > self.pages_per_slot:
            raise MemoryError("out of memory: no free pages in the pool")
        slot = self.free.pop()
        weakref.finalize(state, self.free.append, slot)
        first = slot * self.pages_per_slot
        full = np.full((len(tokens), self.g.cfg.max_blocks_per_seq), -1, dtype=np.int32)
        full[:, :table.shape[1]] = np.where(table >= 0, table + first, -1)
        view = self.g.kv_view()[:, first:first + n]
        return torch.from_numpy(full).to(self.g.dev), view


def _config(shape, c, blocks):
    from paper_2410_21951_b200.binding import make_config
    return make_config(shape, c["batch"], c["nodes"], c["blocks"], blocks, 10, 0, c["rows"])


_CONTEXTS = {}


def _context(model):
    if model not in _CONTEXTS:
        _CONTEXTS[model] = _Context(model)
    return _CONTEXTS[model]


class _State:
    pass


# ---- a case's inputs -------------------------------------------------------------------------------------------------

def _lengths(batch, lo, hi, rng):
    """Lengths spread evenly over [lo, hi], in random order."""
    return rng.permutation(np.linspace(lo, hi, batch).round().astype(np.int32) if batch > 1 else np.array([hi], dtype=np.int32))


def _prefixes(shape, lengths, rng):
    """Phonemes (ids behind the codec ids), then a prompt whose codec ids stay from frame to frame with probability 0.3."""
    out = np.zeros((len(lengths), int(max(lengths))), dtype=np.int32)
    for b, n in enumerate(lengths):
        ph = min(int(rng.integers(40, 121)), int(n) // 2)
        stay = rng.random(n - ph) < 0.3
        stay[0] = False
        jump = rng.integers(0, shape.vocab - 1, size=n - ph)
        out[b, :ph] = shape.vocab + rng.integers(0, shape.n_phonemes, size=ph)
        out[b, ph:n] = jump[np.maximum.accumulate(np.where(stay, 0, np.arange(n - ph)))]
    return out


def _hidden(weights, tokens, gen, dtype):
    """Final hidden states at positions that hold `tokens`: the token's direction and as much of everything else."""
    u = weights["unit"][tokens]
    return (0.7 * u + 0.7 * torch.randn(u.shape, generator=gen, device=u.device)).to(dtype)


def _continue(s, case, rng, gen):
    """A batch whose contexts are in the cache already: K/V rows, the carried hidden state and logits."""
    c, g = s.c, s.c.g
    s.lengths = _lengths(case["batch"], case["ctx_lo"], case["ctx_hi"], rng)
    s.iterations = case.get("iterations", 1)
    s.table, s.view = c.pages(s, [int(n) + case["nodes"] + 5 * s.iterations + 8 for n in s.lengths], int(rng.integers(1 << 31)))
    for layer in s.view:
        layer.normal_(0.0, 0.64, generator=gen)                            # as LayerNorm rows through N(0, 0.02) matrices
    last = torch.from_numpy(rng.integers(0, c.shape.vocab - 1, size=case["batch"])).to(g.dev)
    s.hidden = _hidden(c.weights, last, gen, g.tdtype)
    s.logits = (s.hidden.float() @ c.weights["lm"].T).contiguous()
    s.root = c.weights["succ"][last].cpu().numpy()


def prepare(case, seed):
    rng, gen = np.random.default_rng(seed), torch.Generator(device="cuda").manual_seed(seed)
    if case["kind"] == "fit":
        return _prepare_fit(case, seed, gen)
    s = _State()
    s.kind, s.c = case["kind"], _context(case["model"])
    g, B = s.c.g, case["batch"]
    s.sampling = P.Sampling.make(tau=case.get("tau", 1), temperature=case.get("temperature", 0.0), top_p=case.get("top_p", 1.0), seed=seed)
    if s.kind in ("generate", "prefill"):
        lengths = _lengths(B, case["prefix_lo"], case["prefix_hi"], rng)
        s.lengths = np.ascontiguousarray(lengths, dtype=np.int32)
        s.tokens = _prefixes(s.c.shape, s.lengths, rng)
        more = case["new_tokens"] + case["nodes"] + 8 if s.kind == "generate" else 0
        s.table, s.view = s.c.pages(s, [int(n) + more for n in s.lengths], seed)
        s.view.zero_()
        s.nodes = case.get("nodes", 16)
        if s.kind == "generate":
            s.out, s.out_len = np.zeros((B, case["new_tokens"]), dtype=np.int32), np.zeros(B, dtype=np.int32)
        return s
    _continue(s, case, rng, gen)
    n = s.iterations
    s.accept_len = torch.zeros(n, B, dtype=torch.int32, device=g.dev)
    s.path_tokens = torch.zeros(n, B, P.MAX_PATH, dtype=torch.int32, device=g.dev)
    s.kv_slots = torch.zeros(n, B, P.MAX_PATH, dtype=torch.int64, device=g.dev)
    s.next_root = torch.zeros(n, B, dtype=torch.int32, device=g.dev)
    if s.kind == "steps":
        s.nodes = case["nodes"]
        return s
    trees = [W.random_topology(case["nodes"], 5, int(rng.integers(1 << 31))) for _ in range(B)]
    s.parent, s.rank = np.stack([t.parent for t in trees]), np.stack([t.rank for t in trees])
    succ = s.c.weights["succ"].cpu().numpy()
    tokens = rng.integers(0, s.c.shape.vocab - 1, size=(B, case["nodes"])).astype(np.int32)
    tokens[:, 0] = s.root
    good = rng.random((B, case["nodes"])) < 0.7                            # best candidates: right with this probability
    for b, t in enumerate(trees):
        for i in range(1, case["nodes"]):
            if t.rank[i] == 0 and good[b, i]:
                tokens[b, i] = succ[tokens[b, t.parent[i]]]
    s.candidates = torch.from_numpy(tokens).to(g.dev)
    s.scores = torch.zeros(B, case["nodes"], s.c.shape.vocab, device=g.dev)
    return s


def _prepare_fit(case, seed, gen):
    """Fitting touches the heads only, so the context holds one layer of the model; it is the state's own, since a step
    rewrites the heads in the weight blob."""
    s = _State()
    shape = replace(MODELS[case["model"]][0], n_layers=1, max_pos=64, dtype=case["dtype"])
    c = dict(batch=1, nodes=16, rows=1, blocks=4)
    g = P.Vadusa(shape, _zeros_for(shape, _config(shape, c, 4)), max_batch=1, max_tree_nodes=16, max_blocks_per_seq=4,
                 kv_num_blocks=4, prefill_rows=1)
    info = {t.name.decode(): t for t in P.tensor_infos(g.cfg)}
    s.kind, s.g, s.steps, s.heads = "fit", g, case["steps"], []
    for i in range(shape.n_draft_heads):
        for part in ("w", "b", "u"):
            t = info[f"draft{i}.{part}"]
            raw = g.blob[t.offset:t.offset + t.nbytes].view(g.tdtype if t.is_matrix else torch.float32)
            raw = raw.view(t.rows_padded, t.cols)[:t.rows]
            raw.copy_(torch.randn(t.rows, t.cols, generator=gen, device=g.dev) * 0.02)
            s.heads.append(raw)
    n = shape.vocab - 1
    unit = torch.randn(n, shape.d_model, generator=gen, device=g.dev)
    succ = torch.randperm(n, generator=gen, device=g.dev)
    stream = torch.randint(0, n, (case["tokens"],), generator=gen, device=g.dev)
    s.hidden = _hidden(dict(unit=unit), stream, gen, g.tdtype)
    targets, nxt = [], succ[stream]
    for i in range(shape.n_draft_heads):
        nxt = succ[nxt]
        t = nxt.clone()
        t[max(0, case["tokens"] - 2 - i):] = -1                            # the stream ends: no target
        targets.append(t)
    s.targets = torch.stack(targets, dim=1).to(torch.int32).contiguous()
    s.loss = torch.zeros(case["steps"], 1 + shape.n_draft_heads, device=g.dev)
    g.fit_begin(case["tokens"], lam=0.8, lr=0.002, warmup=40)
    return s


# ---- one pass ----------------------------------------------------------------------------------------------------------

def run(s):
    if s.kind == "fit":
        for i in range(s.steps):
            s.g.fit_step(s.hidden, s.targets, s.loss[i])
        return [s.loss] + s.heads
    g = s.c.g
    if s.kind != "verify":
        s.c.set_tree(s.nodes)                                              # a server keeps one template: nothing to do
    if s.kind == "generate":
        g.generate_host(s.sampling, s.table, s.tokens, s.lengths, s.out.shape[1], s.out, s.out_len)
        return [s.out, s.out_len]
    if s.kind == "prefill":
        g.begin(s.table)
        g.prefill(s.tokens, s.lengths)
        return s.view                                                      # the K/V rows that the pages hold now
    g.begin(s.table, ctx_len=s.lengths)
    g.load_state(s.hidden, s.logits)
    if s.kind == "verify":
        g.set_tree(s.parent, s.rank, per_sequence=True)
        s.c.tree = None
    for i in range(s.iterations):
        g.draft(s.sampling)
        if s.kind == "verify":
            g.verify_step(override=s.candidates, logits_out=s.scores)
        else:
            g.verify_step()
        g.accept_and_commit(s.sampling, accept_len=s.accept_len[i], path_tokens=s.path_tokens[i], kv_slots=s.kv_slots[i],
                            next_root=s.next_root[i])
    return [s.accept_len, s.path_tokens, s.kv_slots, s.next_root] + ([s.scores, s.view] if s.kind == "verify" else [])


# ---- what a pass cannot do without -------------------------------------------------------------------------------------

def _model_work(sh, tokens, context, es, heads=0, logits=0):
    """(bytes, flops) of `tokens` rows through the model, each seeing `context` cached positions on average; every matrix
    is read once.  heads: rows that go through the draft heads; logits: rows that go through the base vocabulary head."""
    layer = 4 * sh.d_model ** 2 + 2 * sh.d_model * sh.d_ffn
    head = sh.n_draft_heads * (sh.d_model ** 2 + sh.vocab * sh.d_model)
    lm = sh.vocab * sh.d_model
    nbytes = es * (sh.n_layers * layer + (head if heads else 0) + (lm if logits else 0))
    flops = 2.0 * (tokens * sh.n_layers * layer + heads * head + logits * lm) + 4.0 * tokens * context * sh.d_model * sh.n_layers
    return nbytes, flops


def work(case):
    sh = MODELS[case["model"]][0]
    if case["kind"] == "fit":
        n = sh.n_draft_heads * (sh.d_model ** 2 + sh.d_model + sh.vocab * sh.d_model)
        es = 2 if case["dtype"] == "bf16" else 4
        rows = case["tokens"] * (sh.d_model * es + 4 * sh.n_draft_heads)
        # a step reads and writes the fp32 heads and both moments, and writes the deployed heads; forward, and twice that backward
        # (no gradient goes to the hidden states: two products for U, one for W)
        per_token = 2.0 * sh.n_draft_heads * (2 * sh.d_model ** 2 + 3 * sh.vocab * sh.d_model)
        return {"bytes": case["steps"] * (n * (24 + es) + rows), "flops": case["steps"] * per_token * case["tokens"]}
    es, B = 2 if sh.dtype == "bf16" else 4, case["batch"]
    kv = 2 * sh.d_model * es * sh.n_layers                                 # K/V bytes of one position
    if case["kind"] in ("generate", "prefill"):
        mean = (case["prefix_lo"] + case["prefix_hi"]) / 2 if B > 1 else case["prefix_hi"]
        nbytes, flops = _model_work(sh, B * mean, mean / 2, es, logits=B)
        nbytes += B * mean * kv
        if case["kind"] == "prefill":
            return {"bytes": nbytes, "flops": flops}
        n = -(-case["new_tokens"] // MEAN_ACCEPTED)                        # iterations
        ctx = mean + case["new_tokens"] / 2
        b, f = _model_work(sh, B * case["nodes"], ctx, es, heads=B, logits=B * case["nodes"])
        return {"bytes": nbytes + n * (b + B * (ctx + case["nodes"]) * kv), "flops": flops + n * f}
    n = case.get("iterations", 1)
    ctx = (case["ctx_lo"] + case["ctx_hi"]) / 2 if B > 1 else case["ctx_hi"]
    b, f = _model_work(sh, B * case["nodes"], ctx, es, heads=B, logits=B * case["nodes"])
    scores = B * case["nodes"] * sh.vocab * 4 if case["kind"] == "verify" else 0
    return {"bytes": n * (b + B * (ctx + case["nodes"]) * kv) + scores, "flops": n * f}


def tolerance(case):
    if case["kind"] == "generate":
        return {"rel": 0.0, "differ": 0.01}                                # token ids; a nearly tied draw may fall the other way
    if case["kind"] == "fit":
        return {"rel": 2e-3}                                               # fp32 sums; a master next to a bf16 boundary is deployed either way
    if MODELS[case["model"]][0].dtype == "fp32":
        return {"rel": 1e-4, "differ": 0.01}
    return {"rel": 1e-2, "differ": 0.01}                                   # bf16 activations through the layers
