"""The work whose speed counts: calls of the tree-verification library as a
decode loop makes them, through the Python binding of the C ABI.

A case is a dict of plain values.  Its "kind" says which entry points a pass
goes through:

  step       one whole verification step of one sequence (verify_step,
             verify_step_typical or verify_step_sampled): tree attention over
             every layer, LM head with its statistics, acceptance, KV-cache
             compaction
  batch      verify_step_batched[_typical] over a ragged batch
  loop       a CUDA graph of verify_step_scheduled steps (tree and prefix
             length chosen on the device)
  attention  tree_attention of one layer, as a model calls it layer by layer
  staged     a model integration: tree_attention per layer, then
             lm_head_stats, greedy_accept and kv_compact
  lm_head    lm_head_stats alone
  walk       spec_sample_accept alone, from given target logits

Inputs: K, V, queries ~ N(0, 1), LM-head weights ~ N(0, 0.02^2), all bf16.
Each hidden row is noise plus a multiple of one vocabulary row, so that its
softmax has one likely token (p from about 0.1 to 0.99) over a broad
background, as a language model's next-token distribution does; the drafts
name that token at one child of a node with the case's match probability and
random tokens elsewhere.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2606_27550_gb300 as tv
from paper_2606_27550_gb300 import synth

TYPICAL_T, TYPICAL_EPS, TYPICAL_ALPHA = tv.PAPER_TYPICAL
ROPE_BASE = 10000.0
LADDER_UP, LADDER_DOWN = 1.5, 2.5  # nats: the hysteretic ladder over the entropy trace
W_STD = 0.02
LARGEST_BYTES = 8.8e9  # the long-context step


# ---------------------------------------------------------------- the cases


def listed():
    mha = {"q_heads": 32, "kv_heads": 32, "head_dim": 128, "d_model": 4096, "vocab": 32000}
    gqa = {"q_heads": 32, "kv_heads": 8, "head_dim": 128, "d_model": 4096, "vocab": 128256}
    return [
        # the smallest step: one small layer, a 7-node binary tree; launches and latency
        {"name": "tiny_step", "kind": "step", "accept": "greedy", "rope": False, "layers": 1, "q_heads": 4,
         "kv_heads": 4, "head_dim": 64, "d_model": 256, "vocab": 1000, "prefix": 128, "tree": "product", "nodes": 7,
         "match": 0.7},
        # one 7B-shaped layer with its LM head, a 26-node tree: the weight stream dominates
        {"name": "layer_step", "kind": "step", "accept": "greedy", "rope": False, "layers": 1, **mha, "prefix": 1024,
         "tree": "product", "nodes": 26, "match": 0.6},
        # the full decode step at long context: the benchmark's default workload
        {"name": "long_step", "kind": "step", "accept": "greedy", "rope": False, "layers": 32, **mha,
         "prefix": 16384, "tree": "product", "nodes": 64, "match": 0.5},
        # the published setting: typical acceptance, all layers of a 7B model at chat length, queries and
        # tree keys rotated by the call; an odd prefix
        {"name": "typical_step", "kind": "step", "accept": "typical", "rope": True, "layers": 32, **mha,
         "prefix": 1023, "tree": "product", "nodes": 40, "match": 0.7},
        # stochastic verification of the same model further into a conversation
        {"name": "sampled_step", "kind": "step", "accept": "sampled", "rope": False, "layers": 32, **mha,
         "prefix": 2051, "tree": "product", "nodes": 26, "match": 0.7},
        # a grouped-query model with a large vocabulary at long context, the largest tree (256 query rows per kv head)
        {"name": "gqa_long_step", "kind": "step", "accept": "greedy", "rope": False, "layers": 32, **gqa,
         "prefix": 8192, "tree": "product", "nodes": 64, "match": 0.6},
        # serving: a ragged batch of eight sequences, each with its own tree and prefix length
        {"name": "ragged_batch", "kind": "batch", "accept": "greedy", "rope": False, "layers": 1, **gqa, "batch": 8,
         "prefix_min": 512, "prefix_max": 8192, "nodes_min": 4, "match": 0.6, "shape_seed": 5},
        # tree switching on the device: 16 steps over the 8-tree bank in one CUDA graph
        {"name": "scheduled_loop", "kind": "loop", "layers": 1, **mha, "prefix": 2048, "steps": 16, "match": 0.6},
        # one layer of a grouped-query model, as the model's forward pass calls it
        {"name": "layer_attention", "kind": "attention", "rope": False, "layers": 4, "q_heads": 32, "kv_heads": 8,
         "head_dim": 128, "prefix": 4096, "tree": "product", "nodes": 64},
        # a model integration over 16 layers: attention layer by layer, then head, acceptance, compaction
        {"name": "staged_pass", "kind": "staged", "rope": True, "layers": 16, **mha, "prefix": 1500,
         "tree": "product", "nodes": 26, "match": 0.6},
        # the head of a large-vocabulary model over one 64-node tree
        {"name": "lm_head_rows", "kind": "lm_head", "rows": 64, "d_model": 4096, "vocab": 128256},
        # the sampling walk over the largest vocabularies
        {"name": "walk_large_vocab", "kind": "walk", "vocab": 150004, "tree": "product", "nodes": 64, "match": 0.6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_heads(rng, nodes):
    while True:
        kv_heads, group = rng.choice([2, 4, 8, 16, 32]), rng.choice([1, 1, 2, 4, 8])
        if kv_heads * group <= 64 and nodes * group <= 256:
            return {"q_heads": kv_heads * group, "kv_heads": kv_heads, "head_dim": rng.choice([64, 128, 128])}


def _draw_tree(rng):
    return {"tree": rng.choice(["product", "product", "chain", "random"]), "nodes": _log_int(rng, 1, 64)}


def _draw_head_shape(rng):
    return {"d_model": rng.choice([256, 520, 1024, 2048, 4096, 4096, 5120]), "vocab": _log_int(rng, 1000, 152064)}


def draw(rng):
    """One more case of the ranges above: head widths 64 and 128, groups 1 to 8,
    prefixes 1 to 32768, 1 to 32 layers, every tree size, vocabularies 1000 to
    152064, the three acceptance rules, with and without the rotary embedding."""
    while True:
        kind = rng.choice(["step", "step", "step", "step", "batch", "loop", "attention", "attention", "staged",
                           "lm_head", "walk"])
        match = round(rng.uniform(0.3, 0.9), 2)
        c = {"kind": kind}
        if kind in ("step", "attention", "staged"):
            c.update(_draw_tree(rng))
            c.update(_draw_heads(rng, c["nodes"]))
            c["rope"] = rng.random() < 0.4
            c["prefix"] = _log_int(rng, 1, 32768)
            if kind == "step":
                c["layers"] = _log_int(rng, 1, 32)
                c.update(_draw_head_shape(rng), match=match, accept=rng.choice(["greedy", "typical", "sampled"]))
            elif kind == "attention":
                c["layers"] = rng.randint(1, 4)
            else:
                c["layers"] = rng.randint(1, 16)
                c.update(_draw_head_shape(rng), match=match)
        elif kind == "batch":
            c.update(_draw_heads(rng, 64))
            c.update(_draw_head_shape(rng), match=match, accept=rng.choice(["greedy", "typical"]))
            lo = _log_int(rng, 1, 2048)
            c.update(rope=rng.random() < 0.4, layers=rng.randint(1, 4), batch=rng.randint(2, 16), prefix_min=lo,
                     prefix_max=_log_int(rng, lo, 16384), nodes_min=rng.choice([1, 4, 16]),
                     shape_seed=rng.randint(0, 10**6))
        elif kind == "loop":
            c.update(_draw_heads(rng, 64))
            c.update(_draw_head_shape(rng), match=match, layers=rng.randint(1, 4), prefix=_log_int(rng, 1, 16384),
                     steps=rng.randint(2, 24))
        elif kind == "lm_head":
            c.update(_draw_head_shape(rng), rows=_log_int(rng, 1, 256))
        else:
            c.update(_draw_tree(rng), vocab=_log_int(rng, 1000, 152064), match=match)
        w = work(c)
        if w["bytes"] <= LARGEST_BYTES and w["flops"] <= 5e11:
            return c


# ---------------------------------------------------------------- shapes


def _parents(tree, nodes, seed):
    if tree == "chain":
        return synth.chain(nodes)
    if tree == "random":
        return synth.random_tree(synth.rng(seed, 11), nodes)
    if nodes == 7:
        return synth.full_tree((2, 2))
    return synth.rank_product_tree(synth.BANK_BRANCHING, nodes)


def _case_tree(case):
    """The case's parent array: part of its shape, the same for every seed."""
    return _parents(case["tree"], case["nodes"], case["nodes"])


def _batch_shape(case):
    """(parents, prefix lengths) of the sequences: part of the case's shape."""
    g = synth.rng(case["shape_seed"], 12)
    trees = [t for t in synth.bank_trees() if len(t) >= case["nodes_min"]]
    parents = [trees[int(g.integers(0, len(trees)))] for _ in range(case["batch"])]
    prefixes = [int(g.integers(case["prefix_min"], case["prefix_max"] + 1)) for _ in range(case["batch"])]
    return parents, prefixes


def _attention_work(layers, q_heads, kv_heads, d, prefix, nodes):
    keys = prefix + nodes
    return {"bytes": layers * (4.0 * kv_heads * keys * d + 4.0 * nodes * q_heads * d),
            "flops": 4.0 * layers * q_heads * d * nodes * keys}


def _head_work(rows, d_model, vocab):
    return {"bytes": 2.0 * vocab * d_model + 2.0 * rows * d_model + 12.0 * rows, "flops": 2.0 * rows * d_model * vocab}


def _sum(*works):
    return {k: float(sum(w[k] for w in works)) for k in ("bytes", "flops")}


def work(case):
    kind = case["kind"]
    if kind == "lm_head":
        return _head_work(case["rows"], case["d_model"], case["vocab"])
    if kind == "walk":
        # the target and draft rows of the one node where the replacement is drawn
        return {"bytes": 8.0 * case["vocab"], "flops": 4.0 * case["vocab"]}
    dims = (case["q_heads"], case["kv_heads"], case["head_dim"])
    if kind == "attention":
        return _attention_work(1, *dims, case["prefix"], case["nodes"])
    if kind == "batch":
        parents, prefixes = _batch_shape(case)
        parts = [_attention_work(case["layers"], *dims, L, len(p)) for p, L in zip(parents, prefixes)]
        rows = sum(len(p) for p in parents)
        # up to 256 rows share one reading of the weights
        reads = -(-rows // 256)
        head = _head_work(rows, case["d_model"], case["vocab"])
        head["bytes"] += (reads - 1) * 2.0 * case["vocab"] * case["d_model"]
        return _sum(*parts, head)
    if kind == "loop":
        # every step reads the prefix and the head's weights; its tree is one of the bank's
        one = _sum(_attention_work(case["layers"], *dims, case["prefix"], 16),
                   _head_work(64, case["d_model"], case["vocab"]))
        return {k: case["steps"] * v for k, v in one.items()}
    w = _sum(_attention_work(case["layers"], *dims, case["prefix"], case["nodes"]),
             _head_work(case["nodes"], case["d_model"], case["vocab"]))
    if case.get("accept") == "sampled":
        w["bytes"] += 4.0 * case["nodes"] * case["vocab"] + 8.0 * case["vocab"]  # the logits, then one node's rows
    return w


def tolerance(case):
    """Against the same in 64 bits, bf16 attention outputs (weights and outputs
    rounded to bf16) are off by 1.9e-3 to 2.9e-3 in the 2-norm and the head's
    32-bit statistics by up to 1.2e-5 (4096 products each); about four times
    that.  Tokens, paths and moved cache rows are exact."""
    if case["kind"] == "walk":
        return "exact"
    if case["kind"] == "lm_head":
        return {"rel": 5e-5, "max": 1e-3}
    return {"rel": 1e-2, "max": 6e-2}


# ---------------------------------------------------------------- inputs


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & (2**62 - 1))
    return g


def _normal(shape, g, std=1.0):
    out = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    out.normal_(0.0, std, generator=g)
    return out


def _cache(case, prefix, nodes, g, room=0):
    shape = (case["layers"], case["kv_heads"], prefix + nodes + room, case["head_dim"])
    rope = ROPE_BASE if case.get("rope") else 0.0
    return tv.KvCache(_normal(shape, g), _normal(shape, g), prefix, rope)


def _hidden(rows, W, g):
    """Final hidden rows: noise plus enough of one vocabulary row to give its token a logit of 9 to 16."""
    vocab, d_model = W.shape
    tok = torch.randint(0, vocab, (rows,), generator=g, device="cuda")
    w = W[tok].float()
    spike = 9.0 + 7.0 * torch.rand((rows, 1), generator=g, device="cuda")
    noise = torch.randn((rows, d_model), generator=g, device="cuda")
    return (noise + spike / w.square().sum(1, keepdim=True) * w).bfloat16(), tok


def _drafts(parent, tok, vocab, match, r):
    """One draft token per node: with probability `match` one child of a node
    (the first ranks most often) names the parent's likely token."""
    n = len(parent)
    drafts = r.integers(0, vocab, size=n).astype(np.int32)
    for u in range(n):
        kids = [c for c in range(n) if parent[c] == u]
        if kids and r.random() < match:
            drafts[kids[min(int(r.geometric(0.6)) - 1, len(kids) - 1)]] = tok[u]
    drafts[0] = 0
    return drafts


def _canonical(bank, parent):
    bank_id, _ = bank.add(parent)
    return bank_id, bank.get(bank_id)[0]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _stats(rows):
    return (torch.zeros(rows, dtype=torch.int32, device="cuda"), torch.zeros(rows, device="cuda"),
            torch.zeros(rows, device="cuda"))


def _workspace(case, rows):
    return tv.make_workspace(tv.tb_workspace_size(rows, case.get("layers", 1), case.get("kv_heads", 1),
                                                  case.get("q_heads", 1), case.get("head_dim", 128),
                                                  case.get("vocab", 1), 0))


def _tree_rows(kv, nodes):
    return {"k": kv.k, "v": kv.v, "k_tree": kv.k[:, :, kv.L:kv.L + nodes], "v_tree": kv.v[:, :, kv.L:kv.L + nodes]}


def _draft_probs(z, g):
    """What the draft heads would have drawn from: near the target, noisier."""
    noise = torch.randn(z.shape, generator=g, device="cuda")
    return torch.softmax(0.8 * z / TYPICAL_T + 0.7 * noise, dim=1)


def _sampling_inputs(parent, z, r, g):
    """(drafts, draft_probs, uniforms) whose decisions under the 64-bit walk are
    not within rounding of a tie."""
    n, vocab = z.shape
    q = _draft_probs(z, g)
    drafts = torch.zeros(n, dtype=torch.int32, device="cuda")
    if n > 1:
        par = _dev(np.asarray(parent[1:], dtype=np.int64))
        drafts[1:] = torch.multinomial(q[par], 1, generator=g)[:, 0].int()
    for _ in range(64):
        unif = r.random(2 * n, dtype=np.float32)
        if _walk(parent, drafts.cpu().numpy(), z, q, unif)[2] > 1e-4:
            break
    return drafts, q, _dev(unif)


def prepare(case, seed):
    kind = case["kind"]
    g, r = _generator(seed, 1), synth.rng(seed, 13)
    s = {"kind": kind}
    if kind == "lm_head":
        s["W"] = _normal((case["vocab"], case["d_model"]), g, W_STD)
        s["hidden"], _ = _hidden(case["rows"], s["W"], g)
        s["stats"] = _stats(case["rows"])
        s["ws"] = _workspace(case, case["rows"])
        s["out"] = dict(zip(("argmax", "top1", "entropy"), s["stats"]))
        return s
    s["bank"] = bank = tv.Bank(32, 0)
    if kind == "walk":
        s["bank_id"], parent = _canonical(bank, _case_tree(case))
        n, vocab = len(parent), case["vocab"]
        z = 1.3 * torch.randn((n, vocab), generator=g, device="cuda")
        tok = torch.randint(0, vocab, (n,), generator=g, device="cuda")
        z[torch.arange(n, device="cuda"), tok] = 9.0 + 7.0 * torch.rand(n, generator=g, device="cuda")
        s["logits"], s["logz_t"] = z, torch.logsumexp(z.double() / TYPICAL_T, 1).float()
        s["drafts"], s["q"], s["unif"] = _sampling_inputs(parent, z, r, g)
        s["scratch"], s["result"] = torch.zeros(vocab, device="cuda"), tv.make_result()
        s["out"] = {"result": s["result"]}
        return s
    if kind == "batch":
        return _prepare_batch(case, s, g, r)
    if kind == "loop":
        return _prepare_loop(case, s, g, r, seed)
    s["bank_id"], parent = _canonical(bank, _case_tree(case))
    n = len(parent)
    s["parent"] = parent
    s["kv"] = kv = _cache(case, case["prefix"], n, g, room=64)
    q_layers = 1 if kind == "attention" else case["layers"]
    q_shape = (q_layers, n, case["q_heads"], case["head_dim"])
    s["attn"] = torch.zeros(q_shape, dtype=torch.bfloat16, device="cuda")
    s["queries"] = _normal(q_shape, g)
    s["ws"] = _workspace(case, n)
    if kind == "attention":
        s["layer"] = case["layers"] - 1
        s["out"] = {"attn": s["attn"], "k_tree": kv.k[s["layer"], :, kv.L:kv.L + n]}
        return s
    s["W"] = _normal((case["vocab"], case["d_model"]), g, W_STD)
    s["hidden"], tok = _hidden(n, s["W"], g)
    s["stats"], s["result"] = _stats(n), tv.make_result()
    s["out"] = {"attn": s["attn"], **dict(zip(("argmax", "top1", "entropy"), s["stats"])), "result": s["result"],
                **_tree_rows(kv, n)}
    if kind == "staged":
        s["layer_q"] = [s["queries"][i:i + 1] for i in range(case["layers"])]
        s["layer_out"] = [s["attn"][i:i + 1] for i in range(case["layers"])]
    s["accept"] = case.get("accept", "greedy")
    if s["accept"] == "sampled":
        s["logits"] = torch.zeros((n + 1, case["vocab"]), device="cuda")
        s["out"]["logits"] = s["logits"][:n]
        z = s["hidden"].float() @ s["W"].float().T
        s["drafts"], s["q"], s["unif"] = _sampling_inputs(parent, z, r, g)
    else:
        s["drafts"] = _dev(_drafts(parent, tok.cpu().numpy(), case["vocab"], case["match"], r))
    return s


def _prepare_batch(case, s, g, r):
    parents, prefixes = _batch_shape(case)
    ids = {}
    for p in parents:
        if len(p) not in ids:
            ids[len(p)] = _canonical(s["bank"], p)
    rows = sum(len(p) for p in parents)
    s["W"] = _normal((case["vocab"], case["d_model"]), g, W_STD)
    s["hidden"], tok = _hidden(rows, s["W"], g)
    tok = tok.cpu().numpy()
    s["stats"], s["seqs"], s["parents"] = _stats(rows), [], []
    results = torch.zeros((len(parents), tv.RESULT_INTS), dtype=torch.int32, device="cuda")
    s["out"] = {**dict(zip(("argmax", "top1", "entropy"), s["stats"])), "results": results}
    r0 = 0
    for i, (p, prefix) in enumerate(zip(parents, prefixes)):
        bank_id, parent = ids[len(p)]
        n = len(parent)
        q = _normal((case["layers"], n, case["q_heads"], case["head_dim"]), g)
        drafts = _drafts(parent, tok[r0:r0 + n], case["vocab"], case["match"], r)
        kv = _cache(case, prefix, n, g, room=64)
        seq = tv.Seq(bank_id, kv, q, _dev(drafts), torch.zeros_like(q), results[i])
        s["seqs"].append(seq)
        s["parents"].append(parent)
        s["out"]["seq%02d" % i] = [seq.attn_out, kv.k[:, :, prefix:prefix + n], kv.v[:, :, prefix:prefix + n]]
        r0 += n
    s["ws"] = _workspace(case, rows)
    s["accept"] = case["accept"]
    return s


def _prepare_loop(case, s, g, r, seed):
    s["rungs"] = [_canonical(s["bank"], t) for t in synth.bank_trees()]
    n_max = max(len(p) for _, p in s["rungs"])
    s["W"] = _normal((case["vocab"], case["d_model"]), g, W_STD)
    s["hidden"], tok = _hidden(n_max, s["W"], g)
    tok = tok.cpu().numpy()
    drafts = np.zeros((len(s["rungs"]), n_max), np.int32)
    for i, (_, parent) in enumerate(s["rungs"]):
        drafts[i, :len(parent)] = _drafts(parent, tok, case["vocab"], case["match"], r)
    s["drafts"] = _dev(drafts)
    s["kv"] = kv = _cache(case, case["prefix"], n_max, g, room=8 * case["steps"])
    q_shape = (case["layers"], n_max, case["q_heads"], case["head_dim"])
    s["queries"], s["attn"] = _normal(q_shape, g), torch.zeros(q_shape, dtype=torch.bfloat16, device="cuda")
    s["trace_host"] = synth.ar1_entropy_trace(seed, case["steps"])
    s["trace"] = _dev(s["trace_host"].astype(np.float32))
    s["policy"] = tv.make_policy(tv.TB_POLICY_HYSTERETIC_LADDER, tv.TB_FEATURE_TRACE, [b for b, _ in s["rungs"]],
                                 a=LADDER_UP, b=LADDER_DOWN, trace=s["trace"])
    s["first_rung"] = 4
    s["start"], s["state"] = tv.make_state(s["first_rung"], kv.L), tv.make_state(s["first_rung"], kv.L)
    s["stats"], s["result"], s["ws"] = _stats(n_max), tv.make_result(), _workspace(case, n_max)
    s["out"] = {"attn": s["attn"], **dict(zip(("argmax", "top1", "entropy"), s["stats"])), "result": s["result"],
                "state": s["state"], "k": kv.k, "v": kv.v}

    def step(flags=0):
        tv.verify_step_scheduled(s["bank"], s["policy"], s["state"], kv, s["queries"], s["hidden"], s["W"],
                                 s["drafts"], s["attn"], *s["stats"], s["result"], s["ws"], flags)

    step(tv.TB_NO_COMPACT)  # once outside the capture, which loads the kernels; leaves the cache as it is
    torch.cuda.synchronize()
    s["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s["graph"]):
        s["state"].copy_(s["start"])
        for _ in range(case["steps"]):
            step()
    return s


# ---------------------------------------------------------------- one pass


def run(s):
    kind = s["kind"]
    if kind == "step":
        if s["accept"] == "greedy":
            tv.verify_step(s["bank"], s["bank_id"], s["kv"], s["queries"], s["hidden"], s["W"], s["drafts"], s["attn"],
                           *s["stats"], s["result"], s["ws"])
        elif s["accept"] == "typical":
            tv.verify_step_typical(s["bank"], s["bank_id"], s["kv"], s["queries"], s["hidden"], s["W"], s["drafts"],
                                   s["attn"], *s["stats"], s["result"], s["ws"], TYPICAL_T, TYPICAL_EPS, TYPICAL_ALPHA)
        else:
            tv.verify_step_sampled(s["bank"], s["bank_id"], s["kv"], s["queries"], s["hidden"], s["W"], s["drafts"],
                                   s["q"], s["unif"], TYPICAL_T, s["attn"], *s["stats"], s["logits"], s["result"],
                                   s["ws"])
    elif kind == "batch":
        if s["accept"] == "greedy":
            tv.verify_step_batched(s["bank"], s["seqs"], s["hidden"], s["W"], *s["stats"], s["ws"])
        else:
            tv.verify_step_batched_typical(s["bank"], s["seqs"], s["hidden"], s["W"], *s["stats"], s["ws"], TYPICAL_T,
                                           TYPICAL_EPS, TYPICAL_ALPHA)
    elif kind == "loop":
        s["graph"].replay()
    elif kind == "attention":
        tv.tree_attention(s["bank"], s["bank_id"], s["kv"], s["queries"], s["attn"], s["ws"], layer_begin=s["layer"],
                          n_layers=1)
    elif kind == "staged":
        for i, (q, out) in enumerate(zip(s["layer_q"], s["layer_out"])):
            tv.tree_attention(s["bank"], s["bank_id"], s["kv"], q, out, s["ws"], layer_begin=i, n_layers=1)
        tv.lm_head_stats(s["hidden"], s["W"], *s["stats"], s["ws"])
        tv.greedy_accept(s["bank"], s["bank_id"], s["drafts"], s["stats"][0], s["W"].shape[0], s["kv"].L, s["result"])
        tv.kv_compact(s["kv"], s["result"])
    elif kind == "lm_head":
        tv.lm_head_stats(s["hidden"], s["W"], *s["stats"], s["ws"])
    else:
        tv.spec_sample_accept(s["bank"], s["bank_id"], s["drafts"], s["logits"], s["logz_t"], s["q"], s["unif"], 0,
                              TYPICAL_T, s["scratch"], s["result"])
    return s["out"]


# ---------------------------------------------------------------- the same in 64 bits


def _depths(parent):
    return synth.depth_of(parent)


def _allowed(parent):
    """[n][n]: key node j is an ancestor of query node i, or i itself."""
    n = len(parent)
    m = np.zeros((n, n), dtype=bool)
    for i in range(n):
        j = i
        while j >= 0:
            m[i, j] = True
            j = int(parent[j])
    return _dev(m)


def _rotate(x, pos):
    """Rotary embedding of x [..., n, d] at positions pos [n]: element i pairs with i + d / 2."""
    d = x.shape[-1]
    inv = ROPE_BASE ** (-2.0 * torch.arange(d // 2, dtype=torch.float64, device="cuda") / d)
    a = pos[:, None] * inv
    lo, hi = x[..., :d // 2], x[..., d // 2:]
    return torch.cat((lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()), -1)


def _exact_attention(k, v, queries, parent, prefix, rope):
    """One layer: k, v bf16 [kv heads][slots][d], queries [n][q heads][d].  Returns the output and the tree's key
    rows (rotated in place in the bf16 cache when rope)."""
    n, q_heads, d = queries.shape
    group = q_heads // k.shape[0]
    q = queries.double().permute(1, 0, 2)
    tree_k = k[:, prefix:prefix + n].double()
    if rope:
        pos = _dev((prefix + _depths(parent)).astype(np.float64))
        q, tree_k = _rotate(q, pos), _rotate(tree_k, pos)
        k[:, prefix:prefix + n] = tree_k.bfloat16()
    out = torch.empty((q_heads, n, d), dtype=torch.float64, device="cuda")
    allow = _allowed(parent)
    for h in range(k.shape[0]):
        kk, vv = k[h, :prefix + n].double(), v[h, :prefix + n].double()
        z = q[h * group:(h + 1) * group].reshape(group * n, d) @ kk.T / math.sqrt(d)
        z = z.view(group, n, prefix + n)
        z[:, :, prefix:].masked_fill_(~allow, -math.inf)
        out[h * group:(h + 1) * group] = (torch.softmax(z, -1).view(group * n, -1) @ vv).view(group, n, d)
    return out.permute(1, 0, 2), tree_k


def _exact_head(hidden, W):
    """(logits, argmax, top1, entropy), 64-bit."""
    z = torch.empty((hidden.shape[0], W.shape[0]), dtype=torch.float64, device="cuda")
    h = hidden.double()
    for v0 in range(0, W.shape[0], 16384):
        z[:, v0:v0 + 16384] = h @ W[v0:v0 + 16384].double().T
    p = torch.softmax(z, 1)
    return z, z.argmax(1).int(), p.max(1).values, -torch.special.xlogy(p, p).sum(1)


def _path(parent, node):
    path = []
    while node >= 0:
        path.append(node)
        node = int(parent[node])
    return path[::-1]


def _accept_path(parent, ok, score):
    """The root path of the deepest node all of whose edges are ok; ties by score, then by id."""
    best, key = 0, None
    for i in range(len(parent)):
        path = _path(parent, i)
        if all(ok[j] for j in path[1:]):
            x = (len(path), sum(score[j] for j in path[1:]), -i)
            if key is None or x > key:
                best, key = i, x
    return _path(parent, best)


def _greedy_path(parent, drafts, argmax):
    ok = [i == 0 or drafts[i] == argmax[parent[i]] for i in range(len(parent))]
    return _accept_path(parent, ok, [0.0] * len(parent))


def _typical_path(parent, drafts, z):
    lp = torch.log_softmax(z / TYPICAL_T, 1)
    p = lp.exp()
    h = -(p * lp).sum(1).cpu().numpy()
    lp = lp.cpu().numpy()
    ok, score = [True], [0.0]
    for i in range(1, len(parent)):
        u = parent[i]
        score.append(float(lp[u, drafts[i]]))
        ok.append(math.exp(score[i]) > min(TYPICAL_EPS, TYPICAL_ALPHA * math.exp(-h[u])))
    return _accept_path(parent, ok, score)


def _walk(parent, drafts, z, q, unif):
    """Speculative sampling in 64 bits: (path, token, distance of the closest decision from a tie)."""
    n, vocab = z.shape
    u, margin = 0, 1.0
    while True:
        r, qu, nxt = torch.softmax(z[u].double() / TYPICAL_T, 0), q[u].double(), -1
        for c in range(u + 1, n):
            if parent[c] != u:
                continue
            t = int(drafts[c])
            ratio = float(r[t] / qu[t])
            margin = min(margin, abs(float(unif[c]) - min(ratio, 2.0)))
            if float(unif[c]) < ratio:
                nxt = c
                break
            r = (r - qu).clamp_min(0)
            r = r / r.sum()
        if nxt < 0:
            break
        u = nxt
    cdf = r.cumsum(0)
    x = float(unif[n + u]) * float(cdf[-1])
    token = min(int((cdf <= x).sum()), vocab - 1)
    near = float((cdf - x).abs().min())
    return _path(parent, u), token, min(margin, 10.0 * near)


def _result(path, bonus, prefix):
    out = torch.full((tv.RESULT_INTS,), -1, dtype=torch.int32)
    out[:4] = torch.tensor([len(path), int(bonus), prefix + len(path), 0], dtype=torch.int32)
    out[4:4 + len(path)] = torch.tensor(path, dtype=torch.int32)
    return out


def _compacted(tree_rows, path):
    """[.., n, d] rows of the tree after the accepted ones moved to the front."""
    out = tree_rows.clone()
    out[..., :len(path), :] = tree_rows[..., path, :]
    return out


def exact(case, seed):
    if work(case)["flops"] > 6e11:
        return None
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "lm_head":
        _, am, t1, en = _exact_head(s["hidden"], s["W"])
        return {"argmax": am, "top1": t1, "entropy": en}
    if kind == "walk":
        parent = s["bank"].get(s["bank_id"])[0]
        path, token, _ = _walk(parent, s["drafts"].cpu().numpy(), s["logits"], s["q"], s["unif"].cpu().numpy())
        return {"result": _result(path, token, 0)}
    rope = bool(case.get("rope"))
    if kind == "attention":
        o, tree_k = _exact_attention(s["kv"].k[s["layer"]], s["kv"].v[s["layer"]], s["queries"][0], s["parent"],
                                     s["kv"].L, rope)
        return {"attn": o[None], "k_tree": tree_k}
    z, am, t1, en = _exact_head(s["hidden"], s["W"])
    am_host = am.cpu().numpy()
    if kind == "batch":
        out, results, r0 = {"argmax": am, "top1": t1, "entropy": en}, [], 0
        for i, (seq, parent) in enumerate(zip(s["seqs"], s["parents"])):
            n = len(parent)
            drafts = seq.draft_tokens.cpu().numpy()
            both = [_exact_attention(seq.kv.k[j], seq.kv.v[j], seq.q[j], parent, seq.kv.L, rope)
                    for j in range(case["layers"])]
            if s["accept"] == "greedy":
                path = _greedy_path(parent, drafts, am_host[r0:r0 + n])
            else:
                path = _typical_path(parent, drafts, z[r0:r0 + n])
            results.append(_result(path, am_host[r0 + path[-1]], seq.kv.L))
            out["seq%02d" % i] = [torch.stack([o for o, _ in both]), _compacted(torch.stack([t for _, t in both]), path),
                                  _compacted(seq.kv.v[:, :, seq.kv.L:seq.kv.L + n], path)]
            r0 += n
        return {**out, "results": torch.stack(results)}
    if kind == "loop":
        kv, rung, L = s["kv"], s["first_rung"], s["kv"].L
        drafts = s["drafts"].cpu().numpy()
        for step in range(case["steps"]):
            _, parent = s["rungs"][rung]
            n = len(parent)
            path = _greedy_path(parent, drafts[rung][:n], am_host)
            if step == case["steps"] - 1:
                # rows of earlier, larger trees stay in the output: only a full-size last tree is known whole
                attn = torch.stack([_exact_attention(kv.k[j], kv.v[j], s["queries"][j][:n], parent, L, False)[0]
                                    for j in range(case["layers"])]) if n == s["queries"].shape[1] else None
                last = _result(path, am_host[path[-1]], L)
            for x in (kv.k, kv.v):
                x[:, :, L:L + n] = _compacted(x[:, :, L:L + n], path)
            L += len(path)
            f = float(np.float32(s["trace_host"][step]))
            rung = min(rung + 1, len(s["rungs"]) - 1) if f < LADDER_UP else max(rung - 1, 0) if f > LADDER_DOWN else rung
        return {"attn": attn, "argmax": am, "top1": t1, "entropy": en, "result": last, "state": None, "k": kv.k,
                "v": kv.v}
    kv, parent = s["kv"], s["parent"]
    n = len(parent)
    v_tree = kv.v[:, :, kv.L:kv.L + n].clone()
    both = [_exact_attention(kv.k[j], kv.v[j], s["queries"][j], parent, kv.L, rope) for j in range(case["layers"])]
    drafts = s["drafts"].cpu().numpy()
    if s["accept"] == "greedy":
        path = _greedy_path(parent, drafts, am_host)
        bonus = am_host[path[-1]]
    elif s["accept"] == "typical":
        path = _typical_path(parent, drafts, z)
        bonus = am_host[path[-1]]
    else:
        path, bonus, _ = _walk(parent, drafts, z, s["q"], s["unif"].cpu().numpy())
    out = {"attn": torch.stack([o for o, _ in both]), "argmax": am, "top1": t1, "entropy": en,
           "result": _result(path, bonus, kv.L), "k": None, "v": None,
           "k_tree": _compacted(torch.stack([t for _, t in both]), path), "v_tree": _compacted(v_tree, path)}
    if s["accept"] == "sampled":
        out["logits"] = z
    return out
