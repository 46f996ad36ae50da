"""Which kernels a layer takes at the lines of the dispatch rules, as the library itself launches them
on a stand-in for the CUDA runtime (no GPU)."""
import pytest

from paper_2412_06355_gb300 import binding

from fake_runtime import Library


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return Library(str(tmp_path_factory.mktemp("fake")))


TWIN, ONE, SHORT = "dendsn_backward_twin_kernel", "dendsn_backward_kernel", "dendsn_backward_twin_short_kernel"


# T, neurons per sample, H*W, samples, K, G, dtype, the backward
@pytest.mark.parametrize("T,N,inner,B,K,G,dtype,want", [
    (8, 4096, 64, 6, 8, 1, "bf16", ONE), (8, 4096, 64, 7, 8, 1, "bf16", TWIN),       # 24576 lanes
    (10, 4096, 64, 32, 8, 1, "bf16", ONE), (10, 4096, 64, 33, 8, 1, "bf16", TWIN),   # 131072
    (9, 4096, 64, 40, 8, 1, "bf16", TWIN), (9, 4096, 64, 40, 8, 1, "f32", ONE), (9, 4096, 64, 40, 8, 2, "f32", TWIN),
    (1, 4096, 64, 300, 8, 1, "bf16", ONE), (1, 4096, 64, 300, 8, 2, "bf16", ONE), (1, 4096, 64, 300, 8, 4, "bf16", TWIN),
    (1, 4096, 64, 600, 8, 2, "bf16", TWIN), (1, 4096, 64, 600, 8, 2, "f32", ONE), (1, 4096, 64, 600, 8, 4, "f32", TWIN),
    (2, 4096, 64, 140, 8, 1, "bf16", ONE), (2, 4096, 64, 150, 8, 1, "bf16", TWIN), (2, 4096, 64, 40, 8, 2, "f32", TWIN),
    (3, 4096, 64, 90, 8, 1, "bf16", ONE), (3, 4096, 64, 100, 8, 1, "bf16", TWIN),
    (4, 4096, 64, 7, 8, 2, "bf16", TWIN), (4, 4096, 64, 6, 8, 2, "bf16", ONE),
    (4, 4096, 4, 100, 8, 2, "bf16", ONE), (8, 4096, 4, 100, 8, 2, "bf16", TWIN), (8, 4096, 4, 100, 8, 2, "f32", ONE),
    (8, 4096, 8, 100, 8, 2, "f32", TWIN), (8, 4096, 4, 100, 16, 2, "f32", TWIN),
    (16, 4096, 4, 100, 16, 2, "f32", ONE), (16, 4096, 4, 100, 16, 1, "f32", TWIN),
    (4, 4096, 4, 10, 4, 1, "f32", ONE), (4, 4096, 4, 10, 4, 2, "f32", SHORT), (4, 4096, 8, 10, 4, 1, "f32", SHORT),
    (6, 4096, 64, 10, 4, 1, "f32", TWIN), (9, 4096, 64, 10, 4, 1, "f32", ONE), (9, 4096, 64, 10, 4, 1, "bf16", TWIN),
])
def test_the_paper_layouts_backward(fake, T, N, inner, B, K, G, dtype, want):
    cfg = binding.make_config(T, B, N, K, G, N // inner, inner, dtype, layout="paper")
    assert fake.launches(cfg)[1] == want
    # never with dL/dS that is aligned for an element but not for a pair
    if want == TWIN:
        assert fake.launches(cfg, gs=(1 << 20) + (2 if dtype == "bf16" else 4))[1] != TWIN


TWF, TWC, STAGED, PLAIN, CHUNK = ("dendsn_forward_twin_kernel", "dendsn_forward_twin_chunk_kernel",
                                  "dendsn_forward_staged_kernel", "dendsn_forward_kernel", "dendsn_forward_chunk_kernel")


@pytest.mark.parametrize("T,N,inner,B,K,G,dtype,psi,want", [
    (6, 4096, 64, 10, 4, 2, "bf16", "mh", TWC), (6, 4096, 64, 10, 4, 2, "f32", "mh", TWF),
    (6, 4000, 50, 10, 8, 2, "f32", "mh", TWF), (6, 4096, 64, 10, 8, 2, "f32", "mh", STAGED),
    (6, 4096, 64, 200, 4, 4, "f32", "mh", TWF), (6, 4096, 64, 260, 4, 4, "f32", "mh", STAGED),
    (6, 4000, 50, 260, 4, 4, "f32", "mh", TWF), (6, 4096, 64, 260, 4, 2, "f32", "mh", TWF),
    (9, 4096, 64, 16, 8, 2, "bf16", "identity", STAGED), (16, 4096, 64, 16, 8, 2, "bf16", "identity", TWC),
    (9, 4096, 64, 40, 8, 2, "bf16", "identity", TWC), (9, 4096, 64, 260, 8, 2, "bf16", "identity", STAGED),
    (9, 4096, 64, 16, 8, 2, "bf16", "mh", TWC), (9, 4000, 50, 16, 8, 2, "bf16", "identity", TWC),
])
def test_the_paper_layouts_forward(fake, T, N, inner, B, K, G, dtype, psi, want):
    cfg = binding.make_config(T, B, N, K, G, N // inner, inner, dtype, psi, layout="paper")
    assert fake.launches(cfg)[0] == want
    if want in (TWF, TWC):                       # spikes or V^s aligned for an element but not for a pair
        A = 1 << 20
        assert fake.launches(cfg, spikes=A + (2 if dtype == "bf16" else 4))[0] not in (TWF, TWC)
        assert fake.launches(cfg, v_out=A + 4)[0] not in (TWF, TWC)
        assert fake.launches(cfg, v_out=A)[0] == want


@pytest.mark.parametrize("T,B,K,want", [
    (12, 6, 16, CHUNK), (12, 7, 16, PLAIN), (12, 64, 8, CHUNK), (12, 65, 8, PLAIN), (8, 6, 16, PLAIN),
    (12, 512, 4, CHUNK), (12, 513, 4, PLAIN), (12, 600, 2, CHUNK),
])
def test_the_forward_in_chunks(fake, T, B, K, want):
    assert fake.launches(binding.make_config(T, B, 4096, K, 1, 64, 64))[0] == want
