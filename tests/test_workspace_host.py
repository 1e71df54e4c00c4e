"""The context's workspace on the host alone: context.cu compiled against a CUDA
runtime that only counts (allocations live on a fake device of a given size, a
stream may be said to be captured).  A buffer that a captured call has used is kept
while its graph may be replayed; one that cannot grow stays, without a wait for the
device or an error text, where the call can go on without it."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_04323_gb300", "csrc")
MB = 1 << 20

FAKE = r"""
#pragma once
#include <cstddef>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
typedef int cudaError_t;
typedef void* cudaStream_t;
typedef void* cudaEvent_t;
enum { cudaSuccess = 0, cudaErrorMemoryAllocation = 2 };
enum cudaStreamCaptureStatus { cudaStreamCaptureStatusNone = 0, cudaStreamCaptureStatusActive = 1 };
enum { cudaMemcpyDeviceToHost = 2 };
static size_t g_room = size_t(1) << 40;
static std::map<void*, size_t> g_live;
static int g_capturing = 0, g_syncs = 0, g_mallocs = 0;
static cudaError_t cudaMalloc(void* out, size_t bytes) {
    ++g_mallocs;
    size_t used = 0;
    for (auto& a : g_live) used += a.second;
    if (used + bytes > g_room) return cudaErrorMemoryAllocation;
    static uintptr_t next = 0;
    void* p = reinterpret_cast<void*>(++next << 8);  // never the same twice
    g_live[p] = bytes;
    std::memcpy(out, &p, sizeof(p));
    return cudaSuccess;
}
static cudaError_t cudaFree(void* p) {
    if (!g_live.erase(p)) std::abort();
    return cudaSuccess;
}
static cudaError_t cudaDeviceSynchronize() { ++g_syncs; return cudaSuccess; }
static cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
static cudaError_t cudaGetLastError() { return cudaSuccess; }
static const char* cudaGetErrorString(cudaError_t) { return "fake"; }
static cudaError_t cudaSetDevice(int) { return cudaSuccess; }
static cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
static cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
static cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
static cudaError_t cudaMemcpyAsync(void*, const void*, size_t, int, cudaStream_t) { return cudaSuccess; }
static cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
static cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
static cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
static cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
static cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
static cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }
"""
HARNESS = r"""
#include "%s/context.cu"
extern "C" {
int t_need(scoot_ctx* c, size_t bytes) { return scoot_workspace(c, bytes, nullptr); }
int t_try(scoot_ctx* c, size_t bytes) { return scoot_workspace_try(c, bytes, nullptr); }
void* t_ws(scoot_ctx* c) { return c->ws; }
int t_lives(void* p) { return g_live.count(p) != 0; }
void t_set(size_t room, int capturing) { g_room = room; g_capturing = capturing; }
int t_syncs() { return g_syncs; }
int t_mallocs() { return g_mallocs; }
size_t t_live_count() { return g_live.size(); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("workspace")
    (d / "cuda_runtime.h").write_text(FAKE)
    (d / "harness.cpp").write_text(HARNESS % CSRC)
    so = str(d / "harness.so")
    subprocess.run([cxx, "-std=c++17", "-D__CUDACC__", "-shared", "-fPIC", f"-I{d}", "-o", so, str(d / "harness.cpp")],
                   check=True)
    lib = ctypes.CDLL(so)
    lib.t_ws.restype = ctypes.c_void_p
    lib.scoot_last_error.restype = ctypes.c_char_p
    lib.t_live_count.restype = ctypes.c_size_t
    return lib


@pytest.fixture
def ctx(lib):
    c = ctypes.c_void_p()
    lib.t_set(ctypes.c_size_t(1 << 40), 0)
    assert lib.scoot_ctx_create(0, ctypes.byref(c)) == 0
    yield c
    lib.t_set(ctypes.c_size_t(1 << 40), 0)
    assert lib.scoot_ctx_destroy(c) == 0
    assert lib.t_live_count() == 0  # everything is given back


def need(lib, c, bytes_, capturing=0, room=1 << 40, kind="t_need"):
    lib.t_set(ctypes.c_size_t(room), capturing)
    r = getattr(lib, kind)(c, ctypes.c_size_t(bytes_))
    lib.t_set(ctypes.c_size_t(1 << 40), 0)
    return r


@pytest.mark.parametrize("kind", ["t_need", "t_try"])
def test_a_captured_buffer_outlives_growth(lib, ctx, kind):
    assert need(lib, ctx, 4 * MB) == 0
    old = lib.t_ws(ctx)
    assert need(lib, ctx, 2 * MB, capturing=1, kind=kind) == (kind == "t_try")
    syncs = lib.t_syncs()
    assert need(lib, ctx, 5 * MB, kind=kind) == (kind == "t_try")
    assert lib.t_ws(ctx) != old and lib.t_lives(ctypes.c_void_p(old)) and lib.t_syncs() == syncs
    held = ctypes.c_int64()
    assert lib.scoot_ctx_workspace_bytes(ctx, ctypes.byref(held)) == 0 and held.value == 12 * MB
    # the new one is in no graph: it goes when it is replaced
    mid = lib.t_ws(ctx)
    assert need(lib, ctx, 9 * MB) == 0
    assert not lib.t_lives(ctypes.c_void_p(mid)) and lib.t_lives(ctypes.c_void_p(old))


def test_a_buffer_of_no_graph_is_freed(lib, ctx):
    assert need(lib, ctx, 4 * MB) == 0
    old, syncs = lib.t_ws(ctx), lib.t_syncs()
    assert need(lib, ctx, 5 * MB, room=6 * MB) == 0  # both would not have fitted
    assert not lib.t_lives(ctypes.c_void_p(old)) and lib.t_syncs() == syncs + 1


def test_no_room_to_double(lib, ctx):
    assert need(lib, ctx, 4 * MB) == 0 and need(lib, ctx, 4 * MB, capturing=1) == 0
    old = lib.t_ws(ctx)
    assert need(lib, ctx, 5 * MB, room=10 * MB) == 0
    assert lib.t_lives(ctypes.c_void_p(old))
    held = ctypes.c_int64()
    lib.scoot_ctx_workspace_bytes(ctx, ctypes.byref(held))
    assert held.value == 9 * MB


def test_an_attempt_that_fails_leaves_everything(lib, ctx):
    assert need(lib, ctx, 4 * MB) == 0
    old, syncs = lib.t_ws(ctx), lib.t_syncs()
    assert need(lib, ctx, 64 * MB, room=32 * MB, kind="t_try") == 0
    assert need(lib, ctx, 64 * MB, capturing=1, kind="t_try") == 0
    assert lib.t_ws(ctx) == old and lib.t_lives(ctypes.c_void_p(old))
    assert lib.t_syncs() == syncs and lib.scoot_last_error(ctx) == b""
    assert need(lib, ctx, 4 * MB) == 0 and lib.t_ws(ctx) == old


def test_refusals(lib, ctx):
    assert need(lib, ctx, 4 * MB) == 0
    mallocs = lib.t_mallocs()
    assert need(lib, ctx, 5 * MB, capturing=1) == -3
    assert lib.t_mallocs() == mallocs  # nothing is allocated during capture
    assert need(lib, ctx, 64 * MB, room=32 * MB) == -2
    assert need(lib, ctx, 4 * MB) == 0  # and the context goes on
