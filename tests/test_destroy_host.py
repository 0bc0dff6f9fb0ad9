"""A graph destroyed while another device is current, on the CPU: the library's
own object files over the model of the CUDA runtime of test_pool_host (two
devices; kernels do nothing, copies to the host bring zeros).  The work that is
waited for, the memory that is freed and the pool that is settled have to be
those of the graph's device, and the caller's device stays current."""
import ctypes
import glob
import os
import shutil
import subprocess

import pytest

from paper_2305_17813_gb300 import build
from test_pool_host import HOLD, MODEL

REST = r"""
#include <cstdlib>
#include <cstring>
extern "C" {
cudaError_t cudaMemcpyAsync(void *to, const void *, size_t n, cudaMemcpyKind kind, cudaStream_t)
{
    if (kind == cudaMemcpyDeviceToHost)
        std::memset(to, 0, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
// what the compiler's host code of a kernel calls: no module is loaded, and a
// launch whose configuration is refused does not happen
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 1; }
}
"""


@pytest.fixture()
def lib(tmp_path):
    build.build()
    src = tmp_path / "model.cpp"
    src.write_text(MODEL + REST)
    out = tmp_path / "libmodel.so"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    # (symbolic: the model's runtime, not one that the process has loaded)
    subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", build.CSRC,
                    "-I", build.INCLUDE, "-I", cuda, str(src), *sorted(glob.glob(os.path.join(build.BUILD, "*.o"))),
                    "-o", str(out)], check=True)
    x = ctypes.CDLL(str(out), mode=os.RTLD_LAZY)
    for f in ("t_held", "t_threshold"):
        getattr(x, f).restype = ctypes.c_uint64
    return x


@pytest.mark.parametrize("kind", ["map", "set"])
def test_destroy_while_another_device_is_current(lib, kind):
    g = ctypes.c_void_p()
    lib.t_device(1)
    create = lib.mk_graph_create if kind == "map" else lib.mk_set_create
    assert create(ctypes.c_uint32(1000), ctypes.c_uint64(1 << 26), ctypes.c_uint32(1), None, None, ctypes.byref(g)) == 0
    held = lib.t_threshold(1) - HOLD
    assert held > 100 << 20
    lib.t_device(0)
    before = [lib.t_syncs(d) for d in (0, 1)]
    destroy = lib.mk_graph_destroy if kind == "map" else lib.mk_set_destroy
    assert destroy(g) == 0
    assert lib.t_current() == 0
    assert lib.t_wrong() == 0  # every block freed with its own device current
    assert lib.t_syncs(1) > before[1] and lib.t_syncs(0) == before[0]
    assert lib.t_threshold(1) == HOLD
