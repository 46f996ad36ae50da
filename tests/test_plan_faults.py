"""Plans and launches when runtime calls fail, on a stand-in for the CUDA runtime (no GPU)."""
import threading

import pytest
import torch

from paper_2412_06355_gb300 import binding

from fake_runtime import Library


@pytest.fixture
def fake(tmp_path):
    return Library(str(tmp_path))


def in_another_thread(f):
    out = []
    t = threading.Thread(target=lambda: out.append(f()))
    t.start()
    t.join()
    return out[0]


def test_a_failed_residency_query_is_not_remembered(fake):
    """The workspace may be sized on one thread and the backward run on another: a plan made while
    a query failed (another tiling, another scratch size) must not outlive the failure."""
    cfg = binding.make_config(4, 64, 131072, 4, 1, 128, 1024, layout="paper")
    fake.lib.fake_fail_queries(2)             # the forward's and the backward's
    first = fake.sizes(cfg)
    now, there = fake.sizes(cfg), in_another_thread(lambda: fake.sizes(cfg))
    assert now == there
    assert first != now                               # the failure did change the tiling


# the chunk forward of 8 float32 compartments, the time-parallel kernels, the twin backward
CFGS = [(16, 64, 4096, 8, 1, {}), (2048, 2, 2, 4, 2, {}), (8, 64, 4096, 8, 1, dict(C=64, inner=64, layout="paper"))]


@pytest.mark.parametrize("T,B,N,K,G,kw", CFGS)
def test_the_shared_memory_opt_in_outlives_no_context(fake, T, B, N, K, G, kw):
    """After a device reset, and from another context of the device, launches that need more than
    48 KB succeed as the first ones did, on the same and on another thread."""
    cfg = binding.make_config(T, B, N, K, G, **kw)
    first = fake.launches(cfg)
    fake.lib.fake_device_reset()
    assert fake.launches(cfg) == first
    fake.lib.fake_device_reset()
    assert in_another_thread(lambda: fake.launches(cfg)) == first
    fake.lib.fake_use_context(1)
    assert fake.launches(cfg) == first
    fake.lib.fake_device_reset()
    fresh = binding.make_config(T, B, N, K, G, theta=0.75, **kw)      # planned anew
    sizes = fake.sizes(fresh)
    assert sizes == fake.sizes(cfg) and fake.launches(fresh) == first


def test_a_failed_opt_in_is_an_error_and_not_remembered(fake):
    cfg = binding.make_config(2048, 2, 2, 4, 2)
    fake.lib.fake_fail_opt_ins(1)
    with pytest.raises(AssertionError):
        fake.launches(cfg)
    assert fake.launches(cfg)[0] == "tp_forward_kernel"


def test_the_bindings_check_follows_the_plan(fake, monkeypatch):
    """The binding checks a workspace against the plan that the library has now, not against the one
    that it made while a query failed."""
    monkeypatch.setattr(binding, "_lib", fake.lib)
    cfg = binding.make_config(4, 64, 131072, 4, 1, 128, 1024, layout="paper")
    fake.lib.fake_fail_queries(2)
    binding._need(cfg, scratch=torch.empty(1 << 26, dtype=torch.uint8))       # planned while they fail
    now = in_another_thread(lambda: binding.dendsn_workspace_size(cfg))[1]
    binding._need(cfg, scratch=torch.empty(now, dtype=torch.uint8))
    with pytest.raises(ValueError, match="scratch"):
        binding._need(cfg, scratch=torch.empty(now - 16, dtype=torch.uint8))
