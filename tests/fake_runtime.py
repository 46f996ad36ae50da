"""The library's host code on a stand-in for the CUDA runtime (c_host/fake_cudart.c): its
objects linked with that in place of cudart, so that plans, dispatch and the handling of failing
runtime calls run without a GPU. Tensors are addresses that nothing reads."""
import ctypes
import os
import re
import subprocess

from paper_2412_06355_gb300 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INCLUDE = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
ADDRESS = 1 << 20                                  # aligned for every access


class Library:
    def __init__(self, directory):
        build.build()
        objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build._sources()]
        if not all(map(os.path.exists, objs)):
            build.build(force=True)
        so = os.path.join(directory, "libdendsn_fake.so")
        fake = os.path.join(directory, "fake_cudart.o")
        subprocess.run(["gcc", "-c", "-fPIC", "-O1", "-I", CUDA_INCLUDE, "-o", fake,
                        os.path.join(HERE, "c_host", "fake_cudart.c")], check=True)
        # -Bsymbolic: the stand-in's functions, not those of a CUDA runtime already loaded
        subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, *objs, fake], check=True)
        P, cfgp = ctypes.c_void_p, ctypes.POINTER(binding.dendsn_config)
        self.lib = lib = ctypes.CDLL(so)
        lib.dendsn_workspace_size.argtypes = [cfgp] + [ctypes.POINTER(ctypes.c_size_t)] * 2
        lib.dendsn_forward.argtypes = [cfgp] + [P] * 10
        lib.dendsn_backward.argtypes = [cfgp] + [P] * 16
        lib.dendsn_unsized_plan_count.restype = ctypes.c_uint64
        lib.fake_launched.restype = ctypes.c_char_p

    def sizes(self, cfg):
        s, w = ctypes.c_size_t(), ctypes.c_size_t()
        assert self.lib.dendsn_workspace_size(cfg, s, w) == 0
        return s.value, w.value

    def launches(self, cfg, mask=None, spikes=ADDRESS, v_out=None, gs=ADDRESS, saved=ADDRESS):
        """The names of the kernels that a forward and a backward launch."""
        A, lib = ADDRESS, self.lib
        n0 = lib.fake_launches()
        assert lib.dendsn_forward(cfg, A, A, A, A, A, mask, spikes, v_out, saved, None) == 0
        assert lib.dendsn_backward(cfg, A, A, A, A, A, mask, gs, None, saved, A, A, A, A, A, A, None) == 0
        names = [lib.fake_launched(i).decode() for i in range(n0, lib.fake_launches())]
        return [re.search(r"(?:dendsn|tp|param)_[a-z_]+_kernel", n).group() for n in names]
