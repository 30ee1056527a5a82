"""Which of a caller's buffers the network's kernels use themselves (csrc/lbm_mlp_buffers.h), on the CPU."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("mlpbuf")
    src, so = d / "rule.cpp", d / "rule.so"
    src.write_text('#include "lbm_mlp_buffers.h"\n'
                   'extern "C" int in_place(int dev, int man, int d, int own, uintptr_t a) { return mlpbuf::in_place(dev, man, d, own, a); }\n'
                   'extern "C" int overlap(uintptr_t a, size_t n, uintptr_t b, size_t m) { return mlpbuf::overlap(a, n, b, m); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_1705_03141_gb300", "csrc"),
                    str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.in_place.argtypes = [ctypes.c_int] * 4 + [ctypes.c_size_t]
    lib.overlap.argtypes = [ctypes.c_size_t] * 4
    return lib


@pytest.mark.parametrize("dev,managed,device,own,addr,ok", [
    (1, 0, 0, 0, 4096, 1), (1, 0, 1, 1, 4100, 1),
    (1, 0, 1, 0, 4096, 0), (1, 0, 0, 1, 4096, 0),  # another device's memory: staged
    (0, 1, 0, 0, 4096, 1), (0, 1, 3, 0, 4096, 1),  # managed memory is reachable from every device
    (0, 0, 0, 0, 4096, 0),                          # host memory
    (1, 0, 0, 0, 4097, 0), (0, 1, 0, 0, 4098, 0),  # not on a word
])
def test_in_place(rule, dev, managed, device, own, addr, ok):
    assert rule.in_place(dev, managed, device, own, addr) == ok


@pytest.mark.parametrize("a,n,b,m,ok", [(0, 100, 100, 10, 0), (100, 10, 0, 100, 0), (0, 101, 100, 10, 1),
                                         (50, 4, 0, 100, 1), (0, 100, 50, 4, 1), (8, 8, 8, 8, 1)])
def test_overlap(rule, a, n, b, m, ok):
    assert rule.overlap(a, n, b, m) == ok
