"""The twin kernels (paper layout, even H*W: two neighbouring neurons per thread).

Per neuron they run the same operations as the one-neuron-per-thread kernels, so on layers
small enough that both layouts are tiled alike every output is compared bit for bit with the
compartments-innermost layer: chunk edges (T below, at and above 4, 6 and 8, every remainder),
two row lanes per warp, a partial last column tile, several lanes per neuron, per-neuron masks,
pairs that straddle nothing (H*W = 2). Layers of 8-compartment lanes take the twin backward only
from 24576 neurons up; those and layers with several rows per thread, whose gradient sums
may be tiled differently, are compared with the oracle.
"""
import pytest
import torch

import oracle
from paper_2412_06355_gb300 import binding, workloads

from parity import check_layer, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")
    binding.load()
    oracle.build()


def run(w, gs_offset=0):
    inp = to_dev(workloads.make_inputs(w, "cpu", with_gv=True))
    cfg = binding.config_of(w)
    p = [inp[k] for k in ("alpha", "xi", "zeta", "kappa")]
    gs = inp["gs"]
    if gs_offset:
        buf = torch.empty(gs.numel() + gs_offset, dtype=gs.dtype, device="cuda")
        gs = buf[gs_offset:].view(gs.shape).copy_(inp["gs"])
    out = {}
    for want_v in (True, False):
        saved, scratch = binding.workspace(cfg)
        s, v = binding.forward(cfg, inp["x"], *p, inp["mask"], want_v=want_v, saved=saved)
        out["s%d" % want_v] = s
        if want_v:
            out["v"] = v
        for gv in (None, inp["gv"]):
            g = binding.backward(cfg, inp["x"], *p, inp["mask"], gs, gv, saved, scratch,
                                 want_beta=want_v)
            out.update({"%s%d%d" % (k, want_v, gv is None): t for k, t in g.items()})
    torch.cuda.synchronize()
    return out


def same(w, a, b):
    """a: the paper layout's outputs, b: the compartments-innermost layer's."""
    assert a.keys() == b.keys()
    for k in a:
        x = workloads.from_paper_layout(a[k], w.N, w.K, w.inner) if k.startswith("gx0") or \
            k.startswith("gx1") else a[k]
        assert torch.equal(x, b[k]), k


def make(T, K, G, dtype, inner, **kw):
    C = {2: 3, 6: 5, 34: 3, 100: 3}[inner]
    return workloads.Workload("twin", T=T, B=3, N=2 * C * inner, K=K, G=G, C=C, inner=inner,
                              dtype=dtype, psi="mh", reset="hard", seed=100 * T + 10 * K + G,
                              ).with_(**kw)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("K,G", [(2, 1), (2, 2), (4, 1), (4, 2), (4, 4), (16, 1)])
@pytest.mark.parametrize("T", [1, 2, 3, 4, 5, 6, 7, 8, 9, 11, 14, 16])
def test_bitwise_the_kinner_layer(T, K, G, dtype):
    inner = [2, 6, 34, 100][(T + K + G) % 4]
    kw = dict(reset="soft" if T % 2 else "hard", residual=T % 3 == 0, stateless=T % 5 == 0,
              mask_p=0.5 if T % 4 == 1 else None, mask_per_neuron=K == 4 and T % 4 == 1,
              psi="identity" if T % 7 == 2 else "mh")
    w = make(T, K, G, dtype, inner, **kw)
    same(w, run(w.with_(layout="paper")), run(w))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_element_aligned_pointers_give_the_same_bits(dtype):
    w = make(6, 4, 2, dtype, 34, layout="paper")
    a, b = run(w), run(w, gs_offset=1)              # dL/dS not aligned for a pair
    for k in a:
        assert torch.equal(a[k], b[k]), k


# 8-compartment lanes from the sizes that take the twin backward; the last two have several
# rows per thread and odd row counts
@pytest.mark.parametrize("T,K,G,dtype,B,C,inner,kw", [
    (4, 8, 2, "bf16", 25, 5, 200, {}),
    (8, 8, 1, "bf16", 25, 5, 200, dict(reset="soft", mask_p=0.5, mask_per_neuron=True)),
    (6, 8, 1, "f32", 25, 5, 200, dict(residual=True)),
    (16, 8, 2, "f32", 25, 10, 100, dict(mask_p=0.5)),
    (16, 16, 1, "bf16", 13, 10, 100, dict(residual=True)),
    (10, 8, 1, "f32", 67, 10, 200, dict(stateless=True)),
    (3, 16, 2, "bf16", 67, 10, 100, {}),
    (5, 8, 4, "bf16", 67, 10, 200, {}),
    (6, 4, 2, "bf16", 9001, 3, 2, {}),
    (9, 2, 1, "bf16", 9001, 2, 6, dict(mask_p=0.5, mask_per_neuron=True)),
])
def test_against_the_oracle(T, K, G, dtype, B, C, inner, kw):
    w = workloads.Workload("twin8", T=T, B=B, N=C * inner, K=K, G=G, C=C, inner=inner, dtype=dtype,
                           psi="mh", reset="hard", layout="paper", seed=7 * T + K).with_(**kw)
    check_layer(w)


# forwards: spikes (by elements) and V^s (by floats) that are not aligned for a pair
@pytest.mark.parametrize("T,dtype,inner", [(6, "bf16", 34), (10, "bf16", 100), (4, "f32", 6)])
@pytest.mark.parametrize("spike_offset,v_offset", [(1, 0), (0, 1), (1, 1)])
def test_element_aligned_outputs_get_the_same_bits(T, dtype, inner, spike_offset, v_offset):
    w = make(T, 4, 2, dtype, inner, layout="paper")
    inp = to_dev(workloads.make_inputs(w, "cpu"))
    cfg = binding.config_of(w)
    p = [inp[k] for k in ("alpha", "xi", "zeta", "kappa")]
    s0, v0 = binding.forward(cfg, inp["x"], *p, None, want_v=True)
    s = torch.empty(s0.numel() + spike_offset, dtype=s0.dtype, device="cuda")[spike_offset:].view(s0.shape)
    v = torch.empty(v0.numel() + v_offset, device="cuda")[v_offset:].view(v0.shape)
    binding.dendsn_forward(cfg, inp["x"], *p, None, s, v)
    assert torch.equal(s, s0) and torch.equal(v, v0)


# layers just beyond the sizes from which rows of a few steps take the twin backward, and from which
# the forward is staged: the same bits per neuron as the compartments-innermost layer
@pytest.mark.parametrize("T,B,K,G,dtype,psi", [
    (2, 150, 8, 1, "bf16", "mh"), (3, 100, 8, 2, "bf16", "mh"), (1, 600, 8, 2, "bf16", "mh"), (1, 300, 8, 4, "f32", "mh"),
    (6, 260, 4, 4, "f32", "mh"), (9, 16, 8, 2, "bf16", "identity"), (9, 260, 8, 2, "bf16", "identity")])
def test_large_layers_bitwise(T, B, K, G, dtype, psi):
    w = workloads.Workload("twinl", T=T, B=B, N=4096, K=K, G=G, C=64, inner=64, dtype=dtype, psi=psi,
                           reset="hard", seed=T)
    out = []
    for layout in ("paper", "kinner"):
        wl = w.with_(layout=layout)
        inp = workloads.make_inputs(wl, "cuda")
        cfg = binding.config_of(wl)
        p = [inp[k] for k in ("alpha", "xi", "zeta", "kappa")]
        saved, scratch = binding.workspace(cfg)
        s, v = binding.forward(cfg, inp["x"], *p, None, want_v=True, saved=saved)
        g = binding.backward(cfg, inp["x"], *p, None, inp["gs"], None, saved, scratch)
        gx = workloads.from_paper_layout(g["gx"], w.N, w.K, w.inner) if layout == "paper" else g["gx"]
        out.append((s, v, gx))
    for a, b in zip(*out):
        assert torch.equal(a, b)
