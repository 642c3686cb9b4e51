"""Objects are given back on their own device, whichever device the calling
thread has current: the C entry points (gr_api.cu) linked against a stand-in of
the CUDA runtime with two devices, which notes what is called on which."""
import ctypes
import os
import subprocess

import pytest

from paper_2303_15762_gb300 import _native as nat
from paper_2303_15762_gb300 import build as gb
from paper_2303_15762_gb300 import scenegen as sg

RUNTIME = r"""
#include <driver_types.h>
#include <cstdlib>
#include <cstring>
#include <string>
static int g_dev = 0;
static std::string g_log;
static void note(const char* what) { g_log += std::string(what) + std::to_string(g_dev) + " "; }
static cudaError_t get(void** p, size_t n) { return (*p = calloc(n ? n : 1, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
extern "C" {
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_dev = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { note("sync"); return cudaSuccess; }
cudaError_t cudaFree(void* p) { note("free"); free(p); return cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { note("free"); free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return get(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return get(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return get(p, n); }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = (cudaMemPool_t)p; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) { memset(a, 0, sizeof *a); a->type = cudaMemoryTypeHost; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
}
"""
VIEW = sg.grating_view(width=4, height=3, spp=1, n_bins=2)


@pytest.fixture(scope="module")
def api(tmp_path_factory):
    d = tmp_path_factory.mktemp("api")
    (d / "runtime.cpp").write_text(RUNTIME)
    try:
        nvcc = gb.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.check_call([nvcc] + gb.ARCH + gb.NVCC_FLAGS + ["-c", os.path.join(gb.CSRC, "gr_api.cu"),
                                                              "-o", str(d / "api.o")])
    # (its own runtime, also where a process has the real one; the kernels' translation units
    # are left out: the entry points under test call none of them)
    subprocess.check_call(["g++", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", cuda, "-o", str(d / "api.so"),
                           str(d / "runtime.cpp"), str(d / "api.o")])
    L = ctypes.CDLL(str(d / "api.so"), mode=os.RTLD_LAZY)
    L.fake_log.restype = ctypes.c_char_p
    return L


def test_frame_is_released_on_its_own_device(api):
    f = ctypes.c_void_p()
    api.cudaSetDevice(0)
    assert api.gr_frame_create(nat.pack_views([VIEW]), 1, None, ctypes.byref(f)) == 0
    api.cudaSetDevice(1)
    api.fake_clear()
    assert api.gr_frame_release(f) == 0
    assert api.fake_log().decode().split() == ["sync0", "free0", "free0"]  # accumulators, counters
    d = ctypes.c_int()
    api.cudaGetDevice(ctypes.byref(d))
    assert d.value == 1
