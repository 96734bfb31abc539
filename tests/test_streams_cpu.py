"""How the host code orders its internal streams, after an error too, on a CUDA runtime that runs nothing (fake_cudart.cpp)."""
import ctypes
import os
import subprocess

import pytest

import paper_2504_02692_b200 as g
from paper_2504_02692_b200 import build as gbuild

HERE = os.path.dirname(os.path.abspath(__file__))
S = 0x77                      # the caller's stream
ADDR = 1 << 41                # device memory is never touched


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "libgptaq_fake.so")
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=compute_100a", "-O0", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", so, *gbuild.sources(), os.path.join(HERE, "fake_cudart.cpp")], check=True)
    lib = ctypes.CDLL(so)
    lib.fake_unordered.argtypes = [ctypes.c_void_p]
    lib.fake_fail_at.argtypes = [ctypes.c_long]
    lib.fake_calls.restype = ctypes.c_long
    for name, (restype, argtypes) in g.SIGNATURES.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = restype, argtypes
    return lib


class Layer:
    def __init__(self, lib, n, m, tokens):
        self.lib, self.n, self.m, self.tokens = lib, n, m, tokens
        self.h = ctypes.c_void_p()
        assert lib.gptaq_create(ctypes.byref(self.h), n, ADDR, lib.gptaq_state_bytes(n), ADDR,
                                lib.gptaq_workspace_bytes(n, m, tokens, 128), S) == g.GPTAQ_OK

    def call(self, name):
        lib, h, n = self.lib, self.h, self.n
        if name == "accumulate":
            return lib.gptaq_accumulate(h, ADDR, ADDR, self.tokens, n, S)
        if name == "factor":
            return lib.gptaq_factor(h, 0.01, S)
        if name == "build_P":
            return lib.gptaq_build_P(h, 0.25, S)
        return lib.gptaq_quantize(h, ADDR, 0, self.m, n, 4, 128, 0, 128, ADDR, ADDR, ADDR, ADDR, S)


CALLS = ["accumulate", "factor", "build_P", "quantize"]


@pytest.mark.parametrize("n,m", [(1416, 5000), (2048, 16), (257, 40), (128, 16)])
@pytest.mark.parametrize("failing", CALLS)
def test_streams_are_joined_after_any_failing_call(lib, n, m, failing):
    """Every runtime call of the step fails once.  What the caller's stream does next (the next call after an error of the
    solve, gptaq_reset after one of the statistics, whose products go on beside the caller's stream) comes after all that
    the internal streams were given."""
    k = 0
    while True:
        k += 1
        lib.fake_fail_at(0)
        lib.fake_reset()
        layer = Layer(lib, n, m, 3000)
        for name in CALLS[:CALLS.index(failing)]:
            assert layer.call(name) == g.GPTAQ_OK
        lib.fake_fail_at(k)
        status = layer.call(failing)
        reached = lib.fake_calls() >= k
        lib.fake_fail_at(0)
        assert (status == g.GPTAQ_ERR_CUDA) == reached, (k, status)
        if failing == "accumulate":
            assert lib.gptaq_reset(layer.h, S) == g.GPTAQ_OK
        assert lib.fake_unordered(S) == 0, (failing, k)
        assert lib.gptaq_destroy(layer.h) == g.GPTAQ_OK
        if not reached:
            break
    assert k > 1
