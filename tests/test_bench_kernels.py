"""The kernels that bench.py says a layer launches are those that the library launches (on a stand-in
for the CUDA runtime, no GPU)."""
import random

import bench
from paper_2412_06355_gb300 import binding, workloads

from fake_runtime import Library


def layers():
    yield from workloads.WORKLOADS.values()
    rng = random.Random(5)
    for _ in range(4000):
        K, G = rng.choice([(1, 1), (2, 1), (2, 2), (4, 1), (4, 2), (4, 4), (8, 1), (8, 2), (8, 4),
                           (16, 1), (16, 2), (16, 4)])
        C, inner = rng.choice([(1, 1), (64, 1), (512, 4), (64, 64), (16, 49), (8, 196), (128, 1024)])
        T = rng.choice([1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 16, 17, 32, 300, 700, 2400, 9000])
        yield workloads.Workload("k", T=T, B=int(4 ** rng.uniform(0, 6)), N=C * inner, K=K, G=G, C=C, inner=inner,
                                 dtype=rng.choice(["f32", "bf16"]), psi=rng.choice(["mh", "mh", "identity"]),
                                 reset="hard", residual=rng.random() < 0.3,
                                 layout=rng.choice(["kinner", "paper", "paper"]))


def test_launched_kernels(tmp_path):
    fake = Library(str(tmp_path))
    for w in layers():
        got = fake.launches(binding.config_of(w))[:2]
        assert list(bench.launched_kernels(w)) == got, w
