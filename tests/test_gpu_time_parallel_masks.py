"""The time-parallel kernels with 16 branches and a mask (two fetches of 8 branches each), against the
oracle; tolerances are the parity tests'."""
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


@pytest.mark.parametrize("T", [300, 1000])
@pytest.mark.parametrize("per_neuron", [False, True])
@pytest.mark.parametrize("layout", ["kinner", "paper"])
def test_sixteen_masked_branches(T, per_neuron, layout):
    w = workloads.Workload("tpm", T=T, B=2, N=12, K=16, G=1, C=3, inner=4, dtype="f32", psi="mh", reset="hard",
                           mask_p=0.5, mask_per_neuron=per_neuron, layout=layout, seed=T)
    assert binding.dendsn_workspace_size(binding.config_of(w))[0] == 0   # the time-parallel path
    check_layer(w)
