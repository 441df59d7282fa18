"""What the library's host side plans and launches, without a GPU: its objects
linked with a stand-in for the CUDA runtime that records launches and keeps
function attributes per device (tests/fake_cuda)."""
import pytest
import torch

import fake_cuda
import paper_2606_27550_gb300 as tv


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
        tv.spec_sample_accept(bank, bid, _zeros(3, torch.int32), logits, _zeros(3), logits, _zeros(6), 5, 0.7, _zeros(V),
                              tv.make_result("cpu"), stream=7)
        (walk,) = fake_cuda.launches(lib)
        assert (walk.device, walk.cluster, walk.grid, walk.stream) == (device, ctas, (ctas, 1, 1), 7)
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
        tv.tree_attention(bank, bid, tv.KvCache(k, k, L), q, q, ws, stream=7)
        attention = fake_cuda.launches(lib)
        # 32 units: clusters of four where 32 of them fit, else the even split and its merge
        assert [x.cluster for x in attention] == ([4] if device == 0 else [1, 1])
        o = [_zeros(R, torch.int32), _zeros(R), _zeros(R)]
        tv.lm_head_stats(_bf16(R, D), _bf16(V, D), *o, ws, stream=7)
        head = fake_cuda.launches(lib)[0]
        assert (head.cluster, head.grid[0]) == (2, 152 if device == 0 else 40)
        bank.close()
