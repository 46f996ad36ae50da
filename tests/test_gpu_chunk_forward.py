"""The forward in chunks of 8 steps (rows of more than 8 steps): whole and ragged last chunks, several
rows per thread, several lanes per neuron, masks fetched a row ahead, a partial column tile and the
paper layout with an odd H*W, against the oracle (spikes, V^s, checkpoints through the backward)."""
import pytest
import torch

import oracle
from paper_2412_06355_gb300 import binding, workloads

from parity import check_layer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")
    binding.load()
    oracle.build()


@pytest.mark.parametrize("T", [9, 10, 11, 12, 13, 14, 15, 16, 25])
@pytest.mark.parametrize("K,G,dtype", [(1, 1, "f32"), (2, 1, "bf16"), (4, 2, "f32"), (8, 1, "bf16"),
                                       (16, 2, "f32")])
def test_lengths(T, K, G, dtype):
    layout = "paper" if dtype == "f32" and T % 2 else "kinner"
    w = workloads.Workload("chunk", T=T, B=5, N=2 * 3 * 21, K=K, G=G, C=3, inner=21, dtype=dtype,
                           psi="mh", reset="soft" if T % 3 else "hard", residual=T == 14,
                           mask_p=0.5 if T % 2 else None, mask_per_neuron=T % 4 == 1,
                           layout=layout, seed=T + 40 * K)
    check_layer(w)


@pytest.mark.parametrize("T,K,G,dtype,layout", [(10, 4, 1, "f32", "kinner"), (12, 8, 2, "bf16", "kinner"),
                                                (17, 4, 2, "f32", "paper")])
def test_several_rows_per_thread(T, K, G, dtype, layout):
    w = workloads.Workload("chunkrows", T=T, B=9001, N=6, K=K, G=G, C=2, inner=3, dtype=dtype,
                           psi="mh", reset="hard", layout=layout, mask_p=0.5, mask_per_neuron=True,
                           seed=T)
    check_layer(w, with_gv=False)
