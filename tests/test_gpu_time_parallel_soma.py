"""The soma of the time-parallel kernels gives the serial recursion's own bits.

With beta 1, 1/2 or 0 the product beta V is exact, so one charge is one float32 addition: plain
float32 additions over Z[t] are the reference, and Z[t] is V^s[t] of the same layer with beta = 0
(hard reset). Tolerance: none, the bits."""
import numpy as np
import pytest
import torch

from paper_2412_06355_gb300 import binding, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA device")
    binding.load()


def potentials(w, inp):
    cfg = binding.config_of(w)
    assert binding.dendsn_workspace_size(cfg)[0] == 0      # the time-parallel path
    p = [inp[k].cuda() for k in ("x", "alpha", "xi", "zeta", "kappa")]
    s, v = binding.forward(cfg, *p, None, want_v=True)
    return s.cpu().numpy(), v.cpu().numpy()


def serial(z, beta, theta, soft):
    v = np.zeros_like(z[0])
    s = np.zeros(z[0].shape, bool)
    out = np.empty_like(z)
    for t in range(z.shape[0]):
        leak = np.where(s, v - np.float32(theta) if soft else np.float32(0), v)
        v = np.float32(beta) * leak + z[t]
        s = v >= np.float32(theta)
        out[t] = v
    return out


def check(T, reset, beta, mean, std, N):
    w = workloads.Workload("soma", T=T, B=2, N=N, K=4, G=2, C=1, inner=N, dtype="f32", psi="mh",
                           reset="hard", beta=0.0, x_mean=mean, x_std=std, seed=T)
    inp = workloads.make_inputs(w, "cpu")
    _, z = potentials(w, inp)
    s, v = potentials(w.with_(reset=reset, beta=beta), inp)
    ref = serial(z, beta, w.theta, reset == "soft")
    assert np.array_equal(v, ref)
    assert np.array_equal(s, (ref >= np.float32(w.theta)).astype(np.float32))


# N: a few neurons (blocks of up to 256 threads: the sweep before the soma leaves warps diverged
# on a ragged horizon) and about 2000 (one warp)
@pytest.mark.parametrize("T", [256, 257, 290, 384, 385, 511])
@pytest.mark.parametrize("reset,beta,mean,std", [("hard", 0.5, 0.3, 1.0), ("soft", 1.0, 0.3, 1.0)])
@pytest.mark.parametrize("N", [3, 1001])
def test_serial_soma(T, reset, beta, mean, std, N):
    check(T, reset, beta, mean, std, N)


# whole and ragged segments; guesses that meet, meet late and never meet (the last pass)
@pytest.mark.parametrize("T", [512, 513, 1000, 2048])
@pytest.mark.parametrize("reset,beta,mean,std", [("hard", 0.5, 0.3, 1.0), ("hard", 1.0, 0.0, 0.02),
                                                 ("soft", 1.0, 0.3, 1.0), ("soft", 1.0, 0.0, 0.02)])
def test_segments(T, reset, beta, mean, std):
    check(T, reset, beta, mean, std, 9)


# the line between the serial loop and the segments, and the last pass: from the first segment on
# (most guesses never meet) or over the few segments of a quiet stretch
@pytest.mark.parametrize("T,N,quiet", [(703, 5, 0), (704, 5, 0), (705, 5, 0), (737, 5, 0), (2400, 5, 0), (705, 1001, 0),
                                       (1000, 5, 300), (2048, 5, 640), (2048, 5, 900)])
@pytest.mark.parametrize("reset,std", [("hard", 0.02), ("soft", 0.02), ("soft", 1.0)])
def test_the_last_pass(T, N, quiet, reset, std):
    w = workloads.Workload("soma", T=T, B=2, N=N, K=4, G=2, C=1, inner=N, dtype="f32", psi="mh",
                           reset="hard", beta=0.0, x_mean=0.3 if quiet else 0.0, x_std=std, seed=T + N)
    inp = workloads.make_inputs(w, "cpu")
    if quiet:
        inp["x"][T - quiet:] *= 1e-3
    _, z = potentials(w, inp)
    s, v = potentials(w.with_(reset=reset, beta=1.0), inp)
    ref = serial(z, 1.0, w.theta, reset == "soft")
    assert np.array_equal(v, ref)
    assert np.array_equal(s, (ref >= np.float32(w.theta)).astype(np.float32))
