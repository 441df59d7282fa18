"""One step of one sequence in every structure the host may enqueue it in
(helpers.STEP_STRUCTURES; test_host_launches.py asserts which one each shape
takes), against the oracle: alone, several behind one another without a wait of
the host, and replayed from a CUDA graph; the sampled step, whose walk follows
either stream, in each structure too."""
import numpy as np
import pytest

import oracle
from helpers import (STAT_TOL, STEP_STRUCTURES, abs_bits, bits, check_attention_fuzz, gap_filtered_hidden, make_case,
                     softmax_rows, structure_id, to_dev)
from paper_2606_27550_gb300 import synth
from test_gpu_rope import THETA, check_rotated_keys

torch = pytest.importorskip("torch")
tv = pytest.importorskip("paper_2606_27550_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    from paper_2606_27550_gb300 import build

    build.build()
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


def _outputs(dev, layers, N, Hq, d):
    return (torch.zeros((layers, N, Hq, d), dtype=torch.bfloat16, device=dev),
            torch.zeros(N, dtype=torch.int32, device=dev), torch.zeros(N, dtype=torch.float32, device=dev),
            torch.zeros(N, dtype=torch.float32, device=dev), tv.make_result(dev))


def _same(a, b):
    return all(torch.equal(x.view(torch.int16) if x.dtype == torch.bfloat16 else x,
                           y.view(torch.int16) if y.dtype == torch.bfloat16 else y) for x, y in zip(a, b))


def _graph(step):
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        step(s)
    return g


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("shape", STEP_STRUCTURES, ids=structure_id)
def test_step_structure(dev, shape, d):
    _, parent, L, layers, Hq, Hkv, D, V, rope = shape
    c = make_case(41 + L + d, parent, L, layers, Hq, Hkv, d, D, V, 0.7)
    bank = tv.Bank(1, 0)
    bid, _ = bank.add(c.parent)
    kd, vd = to_dev(c.k, dev), to_dev(c.v, dev)
    kv = tv.KvCache(kd, vd, L, rope_theta=THETA if rope else 0.0)
    args = (to_dev(c.q, dev), to_dev(c.hidden, dev), to_dev(c.W, dev), to_dev(c.drafts.astype(np.int32), dev))
    ws = tv.make_workspace(tv.tb_workspace_size(c.N, layers, Hkv, Hq, d, V, 0), dev)
    outs = [_outputs(dev, layers, c.N, Hq, d) for _ in range(4)]

    def step(o, flags, stream=None):
        tv.verify_step(bank, bid, kv, *args, *o, ws, flags, stream)

    if not rope:  # (a rotating call rotates the tree keys in place: once)
        for o in outs[:3]:  # behind one another on the stream: same workspace, other outputs
            step(o, tv.TB_NO_COMPACT)
        torch.cuda.synchronize()
        assert _same(outs[0], outs[1]) and _same(outs[0], outs[2])
        for o in outs[3]:
            o.zero_()
        g = _graph(lambda s: step(outs[3], tv.TB_NO_COMPACT, s))
        for _ in range(2):
            g.replay()
        torch.cuda.synchronize()
        assert _same(outs[0], outs[3])
        for o in outs[0]:
            o.zero_()
        assert np.array_equal(bits(kd), c.k) and np.array_equal(bits(vd), c.v)
    step(outs[0], 0)
    torch.cuda.synchronize()
    out, am, t1, en, res = outs[0]
    got = out.float().cpu().numpy()
    ka, path, bonus = oracle.accept(c.parent, c.drafts, c.argmax)
    k_ref = c.k.copy()
    for layer in range(layers):
        if rope:
            ref, k_rot = oracle.tree_attention_rope(c.q[layer], c.k[layer], c.v[layer], L, c.parent, THETA)
            ref_abs, _ = oracle.tree_attention_rope(c.q[layer], c.k[layer], abs_bits(c.v[layer]), L, c.parent, THETA)
            k_ref[layer][:, L:L + c.N] = k_rot
        else:
            ref = oracle.tree_attention(c.q[layer], c.k[layer], c.v[layer], L, c.parent)
            ref_abs = oracle.tree_attention(c.q[layer], c.k[layer], abs_bits(c.v[layer]), L, c.parent)
        check_attention_fuzz(got[layer], ref, ref_abs, f"layer {layer}")
    assert np.array_equal(am.cpu().numpy(), c.argmax)
    assert np.abs(t1.cpu().numpy() - c.top1).max() <= STAT_TOL
    assert np.abs(en.cpu().numpy() - c.entropy).max() <= STAT_TOL
    r = tv.parse_result(res)
    assert (r["accept_len"], r["path"], r["bonus_token"], r["new_L"], r["status"]) == (ka, path, bonus, L + ka, 0)
    k_ref = oracle.kv_compact(k_ref, L, path)
    if rope:
        check_rotated_keys(bits(kd)[:, :, L:L + c.N], k_ref[:, :, L:L + c.N])
        assert np.array_equal(bits(kd)[:, :, :L], c.k[:, :, :L])
    else:
        assert np.array_equal(bits(kd), k_ref)
    assert np.array_equal(bits(vd), oracle.kv_compact(c.v, L, path))
    bank.close()


# one shape of each structure, the LM head's rows few
SAMPLED = [next(s for s in STEP_STRUCTURES if s[0] == want and not s[8]) for want in ("beside", "clusters", "chain", "fork")]


@pytest.mark.parametrize("shape", SAMPLED, ids=structure_id)
def test_sampled_step_structure(dev, shape):
    _, parent, L, layers, Hq, Hkv, D, V, _ = shape
    d, temp = 64, 0.7
    parent = np.asarray(parent, np.int32)
    N = len(parent)
    g = synth.rng(51 + L)
    k, v = synth.gen_kv(51, layers, Hkv, L + N, d, L + N)
    q = synth.gen_q(51, layers, N, Hq, d)
    W = synth.gen_lm_head(51, V, D)
    hidden, am, _, _, logits = gap_filtered_hidden(51, N, W, want_logits=True)
    # draft distributions peaked on three tokens each, against a nearly flat target: most children are rejected
    spikes = np.zeros((N, V))
    for u in range(N):
        spikes[u, g.choice(V, 3, replace=False)] = g.uniform(9.0, 12.0, 3)
    probs = softmax_rows(spikes, 1.0)
    probs = (probs / probs.sum(axis=1, keepdims=True)).astype(np.float32).astype(np.float64)
    draft = np.zeros(N, np.int32)
    for c in range(1, N):
        draft[c] = g.choice(V, p=probs[parent[c]] / probs[parent[c]].sum())
    bank = tv.Bank(1, 0)
    bid, _ = bank.add(parent)
    kv = tv.KvCache(to_dev(k, dev), to_dev(v, dev), L)
    args = (to_dev(q, dev), to_dev(hidden, dev), to_dev(W, dev), to_dev(draft, dev), to_dev(probs.astype(np.float32), dev),
            to_dev(g.random(2 * N).astype(np.float32), dev), temp)
    ws = tv.make_workspace(tv.tb_workspace_size(N, layers, Hkv, Hq, d, V, 0), dev)
    runs = [_outputs(dev, layers, N, Hq, d) for _ in range(4)]
    rows = [torch.zeros((N + 1, V), dtype=torch.float32, device=dev) for _ in range(4)]

    def step(i, stream=None):
        tv.verify_step_sampled(bank, bid, kv, *args, *runs[i][:4], rows[i], runs[i][4], ws, tv.TB_NO_COMPACT, stream)

    for i in range(3):
        step(i)
    graph = _graph(lambda s: step(3, s))
    graph.replay()
    torch.cuda.synchronize()
    for i in (1, 2, 3):
        assert _same(runs[0], runs[i]) and torch.equal(rows[0][:N], rows[i][:N])
    assert np.array_equal(runs[0][1].cpu().numpy(), am)
    assert np.abs(rows[0][:N].cpu().numpy() - logits).max() <= STAT_TOL
    for layer in range(layers):
        ref = oracle.tree_attention(q[layer], k[layer], v[layer], L, parent)
        ref_abs = oracle.tree_attention(q[layer], k[layer], abs_bits(v[layer]), L, parent)
        check_attention_fuzz(runs[0][0][layer].float().cpu().numpy(), ref, ref_abs, f"layer {layer}")
    # the walk of the step is the walk alone on the rows the step wrote
    logz, _ = oracle.tempered_stats(logits, temp)
    res, scratch = tv.make_result(dev), torch.empty(V, dtype=torch.float32, device=dev)
    tv.spec_sample_accept(bank, bid, args[3], rows[0][:N], to_dev(logz.astype(np.float32), dev), args[4], args[5], L, temp,
                          scratch, res)
    torch.cuda.synchronize()
    got, want = tv.parse_result(runs[0][4]), tv.parse_result(res)
    assert (got["accept_len"], got["path"], got["status"]) == (want["accept_len"], want["path"], 0)
    bank.close()
