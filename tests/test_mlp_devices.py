"""The network's host code on a machine with two devices, against a fake CUDA runtime on the CPU.

The fake keeps device memory in host memory tagged with the device that was current when it was allocated, holds
kernel attributes per device, and launches nothing: a launch that asks for more dynamic shared memory
than its kernel is allowed on the current device is refused, and pointers to another device's memory among
x, target, label and y, the first members of k_rows' second argument, are counted.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <utility>
struct Dim3 { unsigned x, y, z; };
struct Attr { int type, device; void *dptr, *hptr; long reserved[8]; };
static int cur = 0, foreign = 0, launches = 0, last = 0;
static std::map<uintptr_t, std::pair<size_t, int>> mem;
static std::map<std::pair<int, const void*>, int> limit;
static Dim3 G, B;
static size_t S;
static void* T;
static int owner(const void* p) {
  auto it = mem.upper_bound((uintptr_t)p);
  if (it == mem.begin()) return -1;
  --it;
  return (uintptr_t)p < it->first + it->second.first ? it->second.second : -1;
}
extern "C" {
void fake_set_device(int d) { cur = d; }
int fake_foreign() { return foreign; }
int fake_launches() { return launches; }
int cudaGetDevice(int* d) { *d = cur; return 0; }
int cudaMalloc(void** p, size_t n) { *p = calloc(1, n); mem[(uintptr_t)*p] = {n, cur}; return 0; }
int cudaFree(void* p) { mem.erase((uintptr_t)p); free(p); return 0; }
int cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(1, n); return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaGetLastError() { const int e = last; last = 0; return e; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { memmove(d, s, n); return 0; }
int cudaMemsetAsync(void* d, int v, size_t n, void*) { memset(d, v, n); return 0; }
int cudaStreamSynchronize(void*) { return 0; }
int cudaPointerGetAttributes(Attr* a, const void* p) {
  const int o = owner(p);
  a->type = o < 0 ? 0 : 2;
  a->device = o < 0 ? 0 : o;
  return 0;
}
int cudaFuncSetAttribute(const void* f, int, int v) { limit[{cur, f}] = v; return 0; }
int __cudaGetKernel(const void** k, const void* f) { *k = f; return 0; }
int __cudaLaunchKernel(const void* k, Dim3, Dim3, void** args, size_t smem, void*) {
  auto it = limit.find({cur, k});
  if (smem > (size_t)(it == limit.end() ? 48 * 1024 : it->second)) return last = 1;
  ++launches;
  for (int k = 0; smem > 0 && k < 4; ++k) {  // k_rows alone takes dynamic shared memory
    const int o = owner(((void**)args[1])[k]);
    foreign += o >= 0 && o != cur;
  }
  return 0;
}
unsigned __cudaPushCallConfiguration(Dim3 g, Dim3 b, size_t s, void* t) { G = g; B = b; S = s; T = t; return 0; }
int __cudaPopCallConfiguration(Dim3* g, Dim3* b, size_t* s, void* t) { *g = G; *b = B; *s = S; *(void**)t = T; return 0; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fakecuda")
    (d / "fake.cpp").write_text(FAKE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    fake, so = str(d / "libfake.so"), str(d / "mlp.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", str(d / "fake.cpp"), "-o", fake], check=True)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                    "-cudart", "none", "-shared", "-o", so,
                    os.path.join(ROOT, "paper_1705_03141_gb300", "csrc", "lbm_mlp.cu"), fake], check=True,
                   capture_output=True)
    m, f = ctypes.CDLL(so), ctypes.CDLL(fake)
    P, i, fl = ctypes.c_void_p, ctypes.c_int, ctypes.c_float
    m.lbm_mlp_create.argtypes = [i] * 6 + [ctypes.c_ulonglong, P, P]
    m.lbm_mlp_forward.argtypes = [P, P, i, P]
    m.lbm_mlp_train_step.argtypes = [P, P, P, P, i, fl, fl, fl, P]
    m.lbm_mlp_free.argtypes = [P]
    m.lbm_mlp_free.restype = None
    f.cudaMalloc.argtypes = [P, ctypes.c_size_t]
    f.cudaFree.argtypes = [P]
    return m, f


N_IN, N_POS, N_CLS, BATCH = 5, 64, 4, 4096  # 32-row tiles: more than 48 KB in inference too


def _create(m):
    h = ctypes.c_void_p()
    assert m.lbm_mlp_create(N_IN, 256, 4, N_POS, N_CLS, BATCH, 0, None, ctypes.byref(h)) == 0
    return h


def _host():
    x, t = np.zeros((BATCH, N_IN), np.float32), np.zeros((BATCH, N_POS), np.float32)
    return x, t, np.zeros(BATCH, np.int32), np.zeros((BATCH, N_POS + N_CLS), np.float32)


def test_each_device_allows_its_kernels_their_shared_memory(lib):
    m, f = lib
    x, t, lab, y = _host()
    for device in (0, 1, 0):
        f.fake_set_device(device)
        h = _create(m)
        before = f.fake_launches()
        assert m.lbm_mlp_forward(h, x.ctypes.data, BATCH, y.ctypes.data) == 0
        assert m.lbm_mlp_train_step(h, x.ctypes.data, t.ctypes.data, lab.ctypes.data, BATCH, 1.0, 0.2, 1e-3, None) == 0
        assert f.fake_launches() == before + 4  # the fused path
        m.lbm_mlp_free(h)


def test_buffers_of_another_device_are_staged(lib):
    m, f = lib
    x, t, lab, y = _host()
    dev = {}
    for device in (0, 1):
        f.fake_set_device(device)
        dev[device] = [ctypes.c_void_p() for _ in range(4)]
        for p, a in zip(dev[device], (x, t, lab, y)):
            assert f.cudaMalloc(ctypes.byref(p), a.nbytes) == 0
    f.fake_set_device(0)
    h = _create(m)
    for a in dev.values():
        assert m.lbm_mlp_forward(h, a[0], BATCH, a[3]) == 0
        assert m.lbm_mlp_train_step(h, a[0], a[1], a[2], BATCH, 1.0, 0.2, 1e-3, None) == 0
    assert f.fake_foreign() == 0
    m.lbm_mlp_free(h)
    for a in dev.values():
        for p in a:
            f.cudaFree(p)
