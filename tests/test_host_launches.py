"""What the library's host side plans and launches, without a GPU: its objects
linked with a stand-in for the CUDA runtime that records launches and keeps
function attributes per device (tests/fake_cuda)."""
import pytest
import torch

import fake_cuda
import paper_2606_27550_gb300 as tv
from helpers import SCHEDULED_HEADS, SCHEDULED_STEPS, SCHEDULED_STRUCTURES, STEP_STRUCTURES, THREAD_STEPS, structure_id
from paper_2606_27550_gb300 import synth
from test_gpu_parity import BESIDE_LM

STREAM = 7


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    return fake_cuda.build_lib(tmp_path_factory.mktemp("fake"))


@pytest.fixture
def lib(fake_path, monkeypatch):
    monkeypatch.setattr(tv, "_lib", None)
    lib = tv.load(fake_path)
    fake_cuda.launches(lib)
    yield lib
    lib.fake_set_device(0)
    lib.fake_limit_clusters(1, 152)


def _zeros(n, dtype=torch.float32):
    return torch.zeros(n, dtype=dtype)


@pytest.mark.parametrize("V,ctas", [(32768, 8), (32769, 16), (150004, 16), (262144, 16), (262145, 1)])
def test_walk_on_every_device_of_a_process(lib, V, ctas):
    """A function attribute set on one device says nothing about the next: the
    16-CTA walk is above the portable cluster size on each of them."""
    for device in (0, 1, 0, 1):
        lib.fake_set_device(device)
        bank = tv.Bank(1, device)
        bid, _ = bank.add([-1, 0, 0])
        logits = _zeros(3 * V).view(3, V)
        tv.spec_sample_accept(bank, bid, _zeros(3, torch.int32), logits, _zeros(3), logits, _zeros(6), 5, 0.7,
                              _zeros(V), tv.make_result("cpu"), stream=STREAM)
        (walk,) = fake_cuda.launches(lib)
        assert (walk.device, walk.cluster, walk.grid, walk.stream) == (device, ctas, (ctas, 1, 1), STREAM)
        bank.close()


def _bf16(*shape):
    return torch.zeros(shape, dtype=torch.bfloat16)


def test_cluster_plans_follow_the_device(lib):
    """What fits one device is no answer for another: the attention's clusters and
    the LM head's CTA pairs are planned with each device's own count."""
    lib.fake_limit_clusters(1, 20)
    H, L, R, V, D = 32, 1500, 200, 64000, 256
    for device in (0, 1, 0):
        lib.fake_set_device(device)
        bank = tv.Bank(1, device)
        bid, _ = bank.add([-1, 0, 0])
        ws = tv.make_workspace(tv.tb_workspace_size(R, 1, H, H, 128, V, device), "cpu")
        k = _bf16(1, H, L + 3, 128)
        q = _bf16(1, 3, H, 128)
        tv.tree_attention(bank, bid, tv.KvCache(k, k, L), q, q, ws, stream=STREAM)
        attention = fake_cuda.launches(lib)
        # 32 units: clusters of four where 32 of them fit, else the even split and its merge
        assert [x.cluster for x in attention] == ([4] if device == 0 else [1, 1])
        o = [_zeros(R, torch.int32), _zeros(R), _zeros(R)]
        tv.lm_head_stats(_bf16(R, D), _bf16(V, D), *o, ws, stream=STREAM)
        head = fake_cuda.launches(lib)[0]
        assert (head.cluster, head.grid[0]) == (2, 152 if device == 0 else 40)
        bank.close()


def _structure(launches):
    """Of one step: "fork" (the LM head on another stream than the caller's), else by
    its attention: "clusters" that leave no merge, "beside" the LM head (on fewer
    SMs than there are), or "chain" (on every SM)."""
    (attention,) = (x for x in launches if "k1_tree_attention_tc" in x.name)
    head = next(x for x in launches if "k2_lm_head" in x.name)
    if head.stream != STREAM:
        assert attention.stream == STREAM and not attention.pdl
        return "fork"
    assert all(x.pdl and x.stream == STREAM for x in launches)
    if "ELb0ELb1E" in attention.name:  # <head_dim, several sequences, clusters>
        assert not any("k1_merge_split" in x.name for x in launches)
        return "clusters"
    return "beside" if attention.grid[0] < 152 else "chain"


class _Step:
    """Uninitialised inputs of one step (nothing reads them)."""

    def __init__(self, N, L_cap, layers, Hq, Hkv, d, D, V):
        self.k = torch.empty((layers, Hkv, L_cap, d), dtype=torch.bfloat16)
        self.q = torch.empty((layers, N, Hq, d), dtype=torch.bfloat16)
        self.hidden, self.W = torch.empty((N, D), dtype=torch.bfloat16), torch.empty((V, D), dtype=torch.bfloat16)
        self.drafts = torch.empty((8, N), dtype=torch.int32)
        self.o = (torch.empty(N, dtype=torch.int32), torch.empty(N), torch.empty(N))
        self.ws = torch.empty(tv.tb_workspace_size(N, layers, Hkv, Hq, d, V, 0), dtype=torch.uint8)


def _launch_step(lib, parent, L, layers, Hq, Hkv, d, D, V, rope):
    bank = tv.Bank(1, 0)
    bid, _ = bank.add(parent)
    s = _Step(len(parent), L + len(parent), layers, Hq, Hkv, d, D, V)
    tv.verify_step(bank, bid, tv.KvCache(s.k, s.k, L, 10000.0 if rope else 0.0), s.q, s.hidden, s.W, s.drafts, s.q, *s.o,
                   tv.make_result("cpu"), s.ws, stream=STREAM)
    bank.close()
    return fake_cuda.launches(lib)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("case", STEP_STRUCTURES, ids=structure_id)
def test_step_structures(lib, case, d):
    """The shapes that the GPU tests run take the structure they are there for."""
    want, parent, L, layers, Hq, Hkv, D, V, rope = case
    launches = _launch_step(lib, parent, L, layers, Hq, Hkv, d, D, V, rope)
    rotates_itself = rope and not any("k0_rope" in x.name for x in launches)
    assert _structure(launches) + ("_rotating" if rotates_itself else "") == want


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("structure", THREAD_STEPS)
def test_thread_step_structures(lib, structure, d):
    trees, *shape = THREAD_STEPS[structure]
    L, layers, Hq, Hkv, D, V = shape
    for parent in trees:
        got = _structure(_launch_step(lib, parent, L, layers, Hq, Hkv, d, D, V, False))
        assert (got == "fork") == (structure == "fork"), (got, len(parent))


def test_steps_beside_the_lm_head(lib):
    grids = []
    for parent, L, layers, Hq, Hkv, D, V in BESIDE_LM:
        launches = _launch_step(lib, parent, L, layers, Hq, Hkv, 128, D, V, False)
        assert _structure(launches) == "beside"
        grids.append(launches[0].grid[0])
    assert grids == [12, 9, 4, 19]


@pytest.mark.parametrize("want,D,V,L0", SCHEDULED_STRUCTURES)
def test_scheduled_step_structures(lib, want, D, V, L0):
    layers, Hq, Hkv, d = SCHEDULED_HEADS
    bank = tv.Bank(8, 0)
    ids = [bank.add(t)[0] for t in synth.bank_trees()]
    s = _Step(64, L0 + SCHEDULED_STEPS * 7 + 72, layers, Hq, Hkv, d, D, V)
    pol = tv.make_policy(tv.TB_POLICY_HYSTERETIC_LADDER, tv.TB_FEATURE_ENTROPY, ids, a=1.0, b=2.0)
    tv.verify_step_scheduled(bank, pol, tv.make_state(0, L0, "cpu"), tv.KvCache(s.k, s.k, 0), s.q, s.hidden, s.W,
                             s.drafts, s.q, *s.o, tv.make_result("cpu"), s.ws, stream=STREAM)
    assert _structure(fake_cuda.launches(lib)) == want
    bank.close()
