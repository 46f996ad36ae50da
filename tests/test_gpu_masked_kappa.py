"""A masked branch whose kappa is not finite (a diverged or an unused branch)."""
import pytest
import torch

from paper_2412_06355_gb300 import binding, workloads

from parity import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")
    binding.load()


def run(w, inp):
    cfg = binding.config_of(w)
    p = [inp[k] for k in ("alpha", "xi", "zeta", "kappa")]
    saved, scratch = binding.workspace(cfg)
    s, v = binding.forward(cfg, inp["x"], *p, inp["mask"], want_v=True, saved=saved)
    return dict(binding.backward(cfg, inp["x"], *p, inp["mask"], inp["gs"], None, saved, scratch), s=s, v=v)


@pytest.mark.parametrize("T", [4, 10, 260, 600])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_a_per_neuron_mask_leaves_the_branch_out(T, bad):
    """Every neuron masks branch 1: the outputs are those of the layer with kappa = 0 there."""
    w = workloads.Workload("mk", T=T, B=2, N=24, K=4, G=2, C=2, inner=12, dtype="f32", psi="mh",
                           reset="hard", mask_p=0.5, mask_per_neuron=True, seed=T)
    inp = to_dev(workloads.make_inputs(w, "cpu"))
    inp["mask"][:, 1] = 0
    zero = dict(inp, kappa=inp["kappa"].clone())
    zero["kappa"][:, 1] = 0.0
    inp["kappa"][:, 1] = bad
    a, b = run(w, inp), run(w, zero)
    for k in a:
        assert torch.equal(a[k], b[k]), k
