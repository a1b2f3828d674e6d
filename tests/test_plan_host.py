"""The host side of ragged plans, on the CPU: the library's own objects linked
against a recording stand-in for the CUDA runtime.

The stand-in holds the runtime to what its documentation promises and no more: a
cudaMemcpy from pageable memory may return before the data are on the device, and
only a synchronisation of its stream (or a later synchronous copy from the
device) ends it; graphs replayed on a non-blocking stream do not wait for the
default stream.  Device memory is host memory; kernels do not run.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2512_10059_gb300 import _lib, build

RUNTIME = r"""
#include <cstdlib>
#include <cstring>
#include <vector>
#include <cuda_runtime_api.h>
struct Copy { void* dst; std::vector<char> bytes; };
static std::vector<Copy> pending;
static long launches, early;  // graph launches; of which while copies were under way
static void land() {
    for (auto& c : pending) memcpy(c.dst, c.bytes.data(), c.bytes.size());
    pending.clear();
}
static int fail_in;  // the launch that fails, counted from here on (0: none)
static cudaError_t last = cudaSuccess;
#define OK return cudaSuccess
extern "C" {
void fake_fail(int launch) { fail_in = launch; }
long fake_pending() { return (long)pending.size(); }
long fake_launches() { return launches; }
long fake_early() { return early; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(void** k, const void* f) { *k = (void*)f; OK; }
cudaError_t __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, void*) {
    return fail_in > 0 && --fail_in == 0 ? last = cudaErrorLaunchOutOfResources : cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
    *g = *b = dim3(1); *m = 0; *(void**)s = nullptr; OK;
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = malloc(n); OK; }
cudaError_t cudaFree(void* p) { free(p); OK; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind kind) {
    if (kind == cudaMemcpyHostToDevice) {
        pending.push_back({d, std::vector<char>((const char*)s, (const char*)s + n)});
    } else {
        land();
        memcpy(d, s, n);
    }
    OK;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); OK; }
cudaError_t cudaMemcpyFromSymbolAsync(void*, const void*, size_t, size_t, cudaMemcpyKind, cudaStream_t) { OK; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); OK; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; OK; }
cudaError_t cudaGetDevice(int* d) { *d = 0; OK; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorName(cudaError_t) { return "error"; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaDriverGetVersion(int* v) { *v = 13000; OK; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; OK; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    memset(p, 0, sizeof(*p));
    strcpy(p->name, "Stand In");
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    OK;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 1; OK; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 1; OK; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; OK; }
cudaError_t cudaEventDestroy(cudaEvent_t) { OK; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { OK; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { OK; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; OK; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)8; OK; }
cudaError_t cudaStreamDestroy(cudaStream_t) { OK; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { if (!s) land(); OK; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { OK; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = (cudaGraph_t)8; OK; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)8; OK; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { ++launches; early += !pending.empty(); OK; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { OK; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { OK; }
}
"""


@pytest.fixture
def host(tmp_path):
    """A fresh load of the plan code over the stand-in (its caches empty)."""
    objs = [os.path.join(build.OUT, f) for f in ("boys_ragged.o", "boys_abi.o")]
    build.build(force=not all(map(os.path.exists, objs)))
    src, so = tmp_path / "runtime.cpp", tmp_path / "plan_host.so"
    src.write_text(RUNTIME)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    # -Bsymbolic: the stand-in's names, not those of a runtime that torch has loaded
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, str(src), *objs,
                    "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    _lib.lib()  # declares SIGNATURES
    for f in ("boys_ragged_plan_create", "boys_ragged_plan_config", "boys_ragged_plan_destroy"):
        getattr(lib, f).restype, getattr(lib, f).argtypes = _lib.SIGNATURES[f]
    for f in ("fake_pending", "fake_launches", "fake_early"):
        getattr(lib, f).restype = ctypes.c_long
    return lib


def _create(lib, flags):
    off, km = np.array([0, 5, 300, 300, 1000], np.int64), np.array([2, 0, 7, 32], np.int32)
    oo = np.zeros(4, np.int64)
    h = ctypes.c_void_p()
    # the data pointers are never dereferenced: no kernel runs
    assert lib.boys_ragged_plan_create(0x1000, off.ctypes.data, km.ctypes.data, 4, 0x1000, oo.ctypes.data, flags,
                                       ctypes.byref(h)) == 0
    b, x, w = ctypes.c_int(), ctypes.c_int(), ctypes.c_int()
    assert lib.boys_ragged_plan_config(h, ctypes.byref(b), ctypes.byref(x), ctypes.byref(w)) == 0
    lib.boys_ragged_plan_destroy(h)
    return b.value, x.value, w.value


def test_tile_table_is_on_the_device_before_a_replay(host, monkeypatch):
    """Neither the autotuner's replays nor the plan that is handed out may start
    while the tile table and its header are still being copied."""
    _create(host, 1)
    assert host.fake_launches() > 0 and host.fake_early() == 0
    assert host.fake_pending() == 0
    monkeypatch.setenv("BOYS_FORCE_CONFIG", "128,1,0")
    assert _create(host, 2) == (128, 1, 0)
    assert host.fake_pending() == 0


def test_stored_shapes_of_former_kernels_are_not_taken(host, tmp_path, monkeypatch):
    """A cache file written when the shapes stood for other kernels (its keys name
    the library's version only) is passed over; one written now is taken."""
    cache = tmp_path / "tune.txt"
    cache.write_text("Stand_In|sm103|152SM|drv13000|lib100|n2^10|seg4|w23.41 256 2 2\n")
    monkeypatch.setenv("BOYS_AUTOTUNE_CACHE", str(cache))
    best = _create(host, 1)
    assert best == (64, 1, 1) and host.fake_launches() > 0  # every shape takes 1 ms here, the first one wins
    lines = cache.read_text().splitlines()
    assert len(lines) == 2 and lines[1].split()[1:] == ["64", "1", "1"]
    cache.write_text(lines[1].replace(" 64 1 1", " 128 1 0") + "\n")
    again = tmp_path / "again.so"
    shutil.copy(host._name, again)
    fresh = ctypes.CDLL(str(again))
    for f in ("boys_ragged_plan_create", "boys_ragged_plan_config", "boys_ragged_plan_destroy"):
        getattr(fresh, f).restype, getattr(fresh, f).argtypes = _lib.SIGNATURES[f]
    fresh.fake_launches.restype = ctypes.c_long
    assert _create(fresh, 1) == (128, 1, 0) and fresh.fake_launches() == 0


def test_a_failed_launch_is_reported(host):
    """boys_eval_ragged on a grouped workspace: two launches for the table, one over it and
    the gated persistent one; whichever fails, the call says so."""
    _lib.lib()
    call = host.boys_eval_ragged
    call.restype, call.argtypes = _lib.SIGNATURES["boys_eval_ragged"]
    off, km, oo = np.array([0, 5, 300], np.int64), np.array([2, 7], np.int32), np.zeros(2, np.int64)
    ws = np.zeros(130, np.complex128)  # 16-byte elements: aligned as a workspace is
    args = (0x1000, off.ctypes.data, km.ctypes.data, 2, 0x1000, oo.ctypes.data, ws.ctypes.data, ws.nbytes, None)
    assert ws.ctypes.data % 16 == 0 and call(*args) == 0
    for launch in (1, 2, 3, 4):
        host.fake_fail(launch)
        assert call(*args) == 4, launch
        assert call(*args) == 0
