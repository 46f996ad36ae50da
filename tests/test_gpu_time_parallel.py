"""The time-parallel kernels (one block per neuron) at the edges of their rules, against the oracle:
the serial and the guessed soma (below and from 512 steps, whole and ragged segments), guesses that
meet late or never (a soft reset and quiet inputs at beta = 0.95, thresholds at and below 0), and
blocks of every size (few neurons: 512 threads; about 2000: one warp, which then scans every
compartment)."""
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


@pytest.mark.parametrize("T,B,C,inner,K,G,kw", [
    (511, 2, 2, 3, 4, 2, {}),
    (512, 2, 2, 3, 4, 2, {}),
    (513, 2, 2, 3, 4, 1, dict(beta=0.95, x_mean=0.1, x_std=0.5, x_density=0.3)),
    (1000, 3, 1, 5, 8, 2, dict(beta=0.95, x_mean=0.1, x_std=0.5, x_density=0.3)),
    (1024, 2, 3, 2, 4, 2, dict(reset="soft", beta=0.95, x_mean=0.1, x_std=0.5)),
    (800, 2, 1, 4, 4, 2, dict(beta=0.95, x_mean=0.0, x_std=0.05)),
    (600, 2, 2, 2, 2, 1, dict(reset="soft", theta=-0.3, beta=0.9)),
    (520, 1, 2, 2, 16, 2, dict(reset="soft", theta=0.0, residual=True, dtype="bf16")),
    (260, 4, 5, 100, 4, 2, dict(layout="paper", mask_p=0.5, mask_per_neuron=True)),
    (300, 2, 10, 100, 4, 1, dict(reset="soft")),
    (256, 1, 64, 16, 8, 4, dict(residual=True, psi="identity")),
    (640, 8, 4, 60, 16, 1, dict(stateless=True)),
])
def test_edges(T, B, C, inner, K, G, kw):
    w = workloads.Workload("tpe", T=T, B=B, N=C * inner, K=K, G=G, C=C, inner=inner, dtype="f32",
                           psi="mh", reset="hard", seed=T + K).with_(**kw)
    assert binding.dendsn_workspace_size(binding.config_of(w))[0] == 0   # the time-parallel path
    check_layer(w)
