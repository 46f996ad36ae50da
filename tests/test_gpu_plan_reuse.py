"""Plans are kept per thread by the configuration's value: a config changed in place, more configs
than are kept, and calls from several threads all get the plan of their own values, and an
undersized tensor is still refused after a larger one of the same config."""
import threading

import pytest
import torch

from paper_2412_06355_gb300 import binding

pytestmark = pytest.mark.gpu


def sizes(T, K, B):
    return binding.dendsn_workspace_size(binding.make_config(T, B, 512, K, 1, 2, 256))


def test_values_decide():
    if not torch.cuda.is_available():
        pytest.fail("needs a CUDA device")
    torch.zeros(1, device="cuda")
    grid = [(T, K, B) for T in (4, 9, 17) for K in (1, 2, 4, 8) for B in (1, 2, 64)]
    first = [sizes(*g) for g in grid]
    for (T, K, B), (saved, scratch) in zip(grid, first):
        assert saved == ((T + 7) // 8 - 1 if T > 8 else 0) * B * 512 * (K + 1) * 4
        assert scratch > 0
    assert [sizes(*g) for g in reversed(grid)] == first[::-1]
    got = []
    th = [threading.Thread(target=lambda: got.append([sizes(*g) for g in grid])) for _ in range(3)]
    [t.start() for t in th]
    [t.join() for t in th]
    assert got == [first] * 3

    cfg = binding.make_config(4, 2, 512, 4, 1, 2, 256)
    p = [torch.zeros(2, 4, device="cuda") for _ in range(4)]
    x = torch.randn(4, 2, 512, 4, device="cuda")
    s, _ = binding.forward(cfg, x, *p[:2], p[2] + 1, p[3] + 1)
    cfg.T = 8                                       # the same object, another configuration
    with pytest.raises(ValueError):
        binding.dendsn_forward(cfg, x, *p[:2], p[2] + 1, p[3] + 1, None, s)
    x8 = torch.cat([x, x])
    s8, _ = binding.forward(cfg, x8, *p[:2], p[2] + 1, p[3] + 1)
    assert s8.shape[0] == 8 and torch.equal(s8[:4], s)
    cfg.K = 3
    with pytest.raises(binding.DendSNError):
        binding.dendsn_workspace_size(cfg)


def test_paper_layout_scratch_stays_within_the_built_in_buffer():
    """The paper layout is tiled by its own kernels' residency; where the compartments-innermost
    layer fits the 8 MiB buffer of dendsn_backward_noalloc, so does the paper one."""
    torch.zeros(1, device="cuda")
    for K in (2, 8, 16):
        for C, inner in ((2048, 2), (1024, 4), (512, 16), (64, 256)):
            for B in (64, 512):
                for T in (4, 6, 8, 16):
                    a, b = (binding.dendsn_workspace_size(binding.make_config(
                        T, B, C * inner, K, 1, C, inner, layout=lay))[1] for lay in ("kinner", "paper"))
                    assert b <= max(a, 8 << 20), (K, C, inner, B, T)
