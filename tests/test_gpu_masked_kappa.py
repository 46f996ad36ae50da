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


@pytest.mark.parametrize("T", [4, 6, 10])
@pytest.mark.parametrize("K,G", [(4, 1), (4, 2)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_a_channel_mask_is_the_same_in_both_layouts(T, K, G, dtype):
    """A channel's kappa m is a product, in the forward and in the backward, whichever kernels run:
    with an infinite kappa the masked channel's potentials and gradients are NaN, the others' not."""
    w = workloads.Workload("mk", T=T, B=3, N=102, K=K, G=G, C=3, inner=34, dtype=dtype, psi="mh",
                           reset="hard", mask_p=0.5, seed=T)
    out = []
    for layout in ("paper", "kinner"):
        inp = to_dev(workloads.make_inputs(w.with_(layout=layout), "cpu"))
        inp["mask"][:] = 1
        inp["mask"][1, 0] = 0
        inp["kappa"][1, 0] = float("inf")
        out.append(run(w.with_(layout=layout), inp))
    a, b = out
    for k in a:
        x = workloads.from_paper_layout(a[k], w.N, w.K, w.inner) if k == "gx" else a[k]
        assert torch.equal(x.isnan(), b[k].isnan()) and torch.equal(x.nan_to_num(), b[k].nan_to_num()), k
    assert a["gx"].isnan().any() and not a["gx"].isnan().all()
