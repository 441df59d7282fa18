"""The LM head of small vocabularies: clusters of CTAs share each vocab tile's
k-blocks (k2_lm_head_split), against the oracle at the sizes where it can go
wrong: every cluster size, uneven shares of the k-blocks, a d_model that is no
multiple of 64, ragged last tiles, one row and the most rows of each plan;
typical mode with its gathers; and a bounded wait that runs out."""
import time

import numpy as np
import pytest

import oracle
from helpers import STAT_TOL, TYPICAL, gap_filtered_hidden, make_case, softmax_rows, to_dev, typical_drafts
from paper_2606_27550_gb300 import synth

torch = pytest.importorskip("torch")
tv = pytest.importorskip("paper_2606_27550_gb300")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    from paper_2606_27550_gb300 import build

    build.build()
    torch.cuda.set_device(0)
    return torch.device("cuda:0")


def _outs(dev, R):
    return (torch.full((R,), -1, dtype=torch.int32, device=dev), torch.empty(R, dtype=torch.float32, device=dev),
            torch.empty(R, dtype=torch.float32, device=dev))


@pytest.mark.parametrize("R,D,V", [
    (1, 4096, 129),      # 8 CTAs a tile; a last tile of one entry
    (26, 1024, 1000),    # 2 (16 k-blocks)
    (17, 1032, 2000),    # 2, uneven: 17 k-blocks, the last one ragged
    (64, 3000, 777),     # 5: 47 k-blocks
    (112, 4096, 300),    # the most rows of two CTAs per SM
    (113, 2048, 300),    # one CTA per SM, 2 CTAs a tile
    (256, 4096, 640),    # the most rows: 4
    (26, 4096, 19456),   # 152 tiles: 2
    (26, 2048, 19457),   # one more: whole tiles
])
def test_small_vocab_parity(dev, R, D, V):
    W = synth.gen_lm_head(R + D + V, V, D)
    hidden, am, t1, en = gap_filtered_hidden(R * 7 + V, R, W)
    got = _outs(dev, R)
    ws = tv.make_workspace(tv.tb_workspace_size(R, 1, 1, 1, 128, V, 0), dev)
    h, w = to_dev(hidden, dev), to_dev(W, dev)
    for _ in range(2):  # the second call finds the counters as the first one left them
        tv.lm_head_stats(h, w, *got, ws)
        torch.cuda.synchronize()
        assert tv.tb_workspace_status(ws) == 0
        assert np.array_equal(got[0].cpu().numpy(), am)
        assert np.abs(got[1].cpu().numpy() - t1).max() <= STAT_TOL
        assert np.abs(got[2].cpu().numpy() - en).max() <= STAT_TOL


@pytest.mark.parametrize("tree,D,V,T", [(7, 4096, 500, 0.7), (5, 1024, 3001, 1.3), (2, 2048, 200, 0.4)])
def test_small_vocab_typical(dev, tree, D, V, T):
    parent = np.asarray(synth.bank_trees()[tree], np.int32)
    N = len(parent)
    b = tv.Bank(1, 0)
    bid, _ = b.add(parent)
    W = synth.gen_lm_head(N + V, V, D)
    hidden, am, t1, en = gap_filtered_hidden(N * 3 + V, N, W)
    logits = synth.bf16_bits_to_f32(hidden).astype(np.float64) @ synth.bf16_bits_to_f32(W).astype(np.float64).T
    drafts = typical_drafts(300 + N, parent, logits, T, *TYPICAL[1:])
    lz, et = oracle.tempered_stats(logits, T)
    got = _outs(dev, N)
    g_lz, g_et, g_dl = (torch.zeros(N, dtype=torch.float32, device=dev) for _ in range(3))
    ws = tv.make_workspace(tv.tb_workspace_size(N, 1, 1, 1, 128, V, 0), dev)
    tv.lm_head_stats_typical(b, bid, to_dev(hidden, dev), to_dev(W, dev), T, to_dev(drafts.astype(np.int32), dev), *got,
                             g_lz, g_et, g_dl, ws)
    torch.cuda.synchronize()
    assert tv.tb_workspace_status(ws) == 0
    assert np.array_equal(got[0].cpu().numpy(), am)
    assert np.abs(got[1].cpu().numpy() - t1).max() <= STAT_TOL and np.abs(got[2].cpu().numpy() - en).max() <= STAT_TOL
    assert np.abs(g_lz.cpu().numpy() - lz).max() <= STAT_TOL and np.abs(g_et.cpu().numpy() - et).max() <= STAT_TOL
    want = np.array([0.0] + [logits[parent[j], drafts[j]] for j in range(1, N)])
    assert np.abs(g_dl.cpu().numpy() - want)[1:].max(initial=0.0) <= STAT_TOL
    b.close()


def test_small_vocab_logit_rows(dev):
    """The rows a sampled step writes: every entry, nothing past them."""
    parent, L, H, d, D, V = synth.bank_trees()[4], 40, 2, 64, 2048, 777
    c = make_case(21, parent, L, 1, H, H, d, D, V, 0.7)
    N = c.N
    b = tv.Bank(1, 0)
    bid, _ = b.add(c.parent)
    kv = tv.KvCache(to_dev(c.k, dev), to_dev(c.v, dev), L)
    g = synth.rng(22)
    q = to_dev(softmax_rows(g.standard_normal((N, V)), 1.0).astype(np.float32), dev)
    unif = to_dev(g.random(2 * N).astype(np.float32), dev)
    logits = torch.full((N + 1, V), 7.0, dtype=torch.float32, device=dev)
    got, res = _outs(dev, N), tv.make_result(dev)
    out = torch.empty((1, N, H, d), dtype=torch.bfloat16, device=dev)
    ws = tv.make_workspace(tv.tb_workspace_size(N, 1, H, H, d, V, 0), dev)
    tv.verify_step_sampled(b, bid, kv, to_dev(c.q, dev), to_dev(c.hidden, dev), to_dev(c.W, dev),
                           to_dev(c.drafts.astype(np.int32), dev), q, unif, 0.7, out, *got, logits, res, ws)
    torch.cuda.synchronize()
    want = synth.bf16_bits_to_f32(c.hidden).astype(np.float64) @ synth.bf16_bits_to_f32(c.W).astype(np.float64).T
    assert np.abs(logits[:N].cpu().numpy() - want).max() <= STAT_TOL
    assert (logits[N] == 7.0).all()  # the walk's scratch row, unused at this vocabulary
    assert np.array_equal(got[0].cpu().numpy(), c.argmax)
    b.close()


def test_small_vocab_timeout_is_reported_and_next_call_recovers(dev):
    """Every CTA of a cluster gives up and meets the others at the cluster's barriers."""
    R, D, V = 26, 4096, 1000
    W = synth.gen_lm_head(9, V, D)
    hidden, am, t1, _ = gap_filtered_hidden(10, R, W)
    h, w = to_dev(hidden, dev), to_dev(W, dev)
    o = _outs(dev, R)
    t0 = time.time()
    tv.lm_head_stats_noalloc(h, w, *o, flags=tv.TB_DEBUG_EXPIRE_WAIT)
    assert tv.lm_head_stats_noalloc_status() == tv.TB_ETIMEOUT
    assert time.time() - t0 < 20.0
    assert o[0].cpu().tolist() == [-1] * R
    tv.lm_head_stats_noalloc(h, w, *o)
    assert tv.lm_head_stats_noalloc_status() == tv.TB_OK
    assert np.array_equal(o[0].cpu().numpy(), am) and np.abs(o[1].cpu().numpy() - t1).max() <= STAT_TOL
