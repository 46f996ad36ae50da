"""Plans when runtime calls fail, on a stand-in for the CUDA runtime (no GPU)."""
import threading

import pytest

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
