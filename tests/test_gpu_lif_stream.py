"""The LIF backward of long rows of large layers (at least 8 steps, 524288 neurons), against the oracle:
whole and ragged last chunks, both vector widths, both dtypes, resets and dL/dV."""
import pytest
import torch

import oracle
from paper_2412_06355_gb300 import binding

from test_gpu_lif import check_lif

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")
    binding.load()
    oracle.build()


@pytest.mark.parametrize("T,N,kw", [
    (8, 131072, {}), (9, 131072, dict(dtype="bf16")), (15, 131073, dict(reset="soft")),
    (17, 131075, dict(dtype="bf16", detach=True)), (12, 131072, dict(with_gv=False, reset="soft")),
])
def test_long_rows_of_large_layers(T, N, kw):
    assert check_lif(T, 4, N, seed=T, **kw) > 0.0
