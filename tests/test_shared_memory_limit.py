"""Layers whose launches need just about the shared memory that a block has without an opt-in
(48 KB, a kernel's static arrays included), on a stand-in for the CUDA runtime (no GPU), and with
values against the oracle on one."""
import pytest
import torch

import oracle
from paper_2412_06355_gb300 import binding, workloads

from fake_runtime import Library


def test_every_time_parallel_horizon_is_launched(tmp_path):
    fake = Library(str(tmp_path))
    for K, G in [(1, 1), (2, 1), (2, 2), (4, 1), (4, 2), (8, 1), (8, 2), (16, 1), (16, 4)]:
        for T in range(256, 48 * 1024 // (4 * (K + 2)) + 64, 32):
            for B in (1, 700):
                names = fake.launches(binding.make_config(T, B, 2, K, G))
                assert names[0] in ("tp_forward_kernel", "dendsn_forward_kernel", "dendsn_forward_chunk_kernel")


@pytest.mark.gpu
@pytest.mark.parametrize("T,K,G", [(2048, 1, 1), (1744, 2, 1), (1344, 4, 1), (928, 8, 1), (576, 16, 1)])
def test_values_at_the_limit(T, K, G):
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")
    binding.load()
    oracle.build()
    from parity import check_layer
    w = workloads.Workload("smem", T=T, B=1, N=3, K=K, G=G, C=1, inner=3, dtype="f32", psi="mh",
                           reset="hard", seed=T)
    check_layer(w)
