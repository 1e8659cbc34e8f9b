"""Which calls may read their inputs before the preceding grid is complete (csrc/early_start.cu), on the CPU: the file is
compiled against a stand-in for the few runtime calls it makes, which answers with the capture state that a test sets."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2511_02647_b200", "csrc")

STAND_IN = r"""
#include "common.cuh"
static unsigned long long g_capture;                  // id of the capture under way, 0: none
static cudaGraphNode_t g_deps[4];
static size_t g_n;
extern "C" cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus *st, unsigned long long *id, cudaGraph_t *,
                                                const cudaGraphNode_t **, size_t *)
{
    *st = g_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    *id = g_capture;
    return cudaSuccess;
}
extern "C" cudaError_t cudaStreamGetCaptureInfo_v3(cudaStream_t, cudaStreamCaptureStatus *st, unsigned long long *id, cudaGraph_t *,
                                                   const cudaGraphNode_t **deps, const cudaGraphEdgeData **, size_t *n)
{
    *st = g_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    *id = g_capture;
    *deps = g_deps; *n = g_n;
    return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
using namespace fedattn;
extern "C" void set_capture(unsigned long long id, size_t n, size_t a, size_t b)
{
    g_capture = id; g_n = n; g_deps[0] = (cudaGraphNode_t)a; g_deps[1] = (cudaGraphNode_t)b;
}
static EarlyStart g_es;
// a call that reads [in, in + 16) and writes [out, out + 16): 1 when it may read early
extern "C" int start(size_t stream, size_t in, size_t out)
{
    const MemRange i = {(void *)in, 16}, o = {(void *)out, 16};
    g_es = early_start(0, (cudaStream_t)stream, &i, 1, &o, 1);
    return g_es.early;
}
extern "C" int end(int e) { return early_start_end(g_es, (cudaError_t)e); }
"""


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    tmp_path = tmp_path_factory.mktemp("early_start")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src, so = tmp_path / "stand_in.cpp", tmp_path / "early.so"
    src.write_text(STAND_IN)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", cuda,
                           "-x", "c++", str(src), os.path.join(CSRC, "early_start.cu"), "-o", str(so)])
    return so


@pytest.fixture
def lib(built, tmp_path):
    lib = C.CDLL(shutil.copy(built, tmp_path / "early.so"))      # (a record of its own)
    lib.set_capture.argtypes = [C.c_ulonglong, C.c_size_t, C.c_size_t, C.c_size_t]
    lib.start.argtypes = [C.c_size_t] * 3
    return lib


def test_calls_of_one_stream(lib):
    s = 0x100
    assert lib.start(s, 0x1000, 0x2000) == 0                     # nothing known yet
    assert lib.start(s, 0x3000, 0x4000) == 1
    assert lib.start(s, 0x4008, 0x5000) == 0                     # reads what the call before writes
    assert lib.start(s, 0x3000, 0x6000) == 1


def test_captured_calls_of_one_stream(lib):
    s = 0x100

    def call(dep, node, i, o):
        lib.set_capture(7, 1 if dep else 0, dep, 0)
        early = lib.start(s, i, o)
        lib.set_capture(7, 1, node, 0)
        lib.end(0)
        return early

    assert call(0, 0xa, 0x1000, 0x2000) == 0
    assert call(0xa, 0xb, 0x3000, 0x4000) == 1
    assert call(0xb, 0xc, 0x2008, 0x5000) == 0                   # reads what an earlier call writes
    assert call(0xc, 0xd, 0x3000, 0x6000) == 1


@pytest.mark.parametrize("deps", [(0xa, 0xb), (0xb, 0xa), (0xb,), ()])
def test_captured_call_behind_another_branch_waits_first(lib, deps):
    """Branch 1 writes 0x8000 (node b); branch 2, whose record knows only its own call (node a), joins it and reads that."""
    one, two = 0x100, 0x200
    lib.set_capture(7, 0, 0, 0)
    assert lib.start(two, 0x1000, 0x2000) == 0
    lib.set_capture(7, 1, 0xa, 0)
    lib.end(0)
    lib.set_capture(7, 0, 0, 0)
    assert lib.start(one, 0x3000, 0x8000) == 0
    lib.set_capture(7, 1, 0xb, 0)
    lib.end(0)
    lib.set_capture(7, len(deps), *(deps + (0, 0))[:2])
    assert lib.start(two, 0x8000, 0x9000) == 0
    lib.set_capture(7, 1, 0xc, 0)
    lib.end(0)
    assert lib.start(two, 0x3000, 0xb000) == 1                   # behind the call that waited


def test_captured_call_whose_node_is_unknown_is_followed_by_one_that_waits(lib):
    s = 0x100
    lib.set_capture(7, 0, 0, 0)
    lib.start(s, 0x1000, 0x2000)                                 # (its launch failed: no end)
    assert lib.start(s, 0x3000, 0x4000) == 0


@pytest.mark.parametrize("capture", [0, 7])
def test_call_that_was_not_launched_vouches_for_nothing(lib, capture):
    """The call behind it must not start early on the word of a call that was to wait and never ran."""
    s = 0x100
    lib.set_capture(capture, 0, 0, 0)
    lib.start(s, 0x1000, 0x2000)
    lib.set_capture(capture, 1, 0xa, 0)
    assert lib.end(0) == 0
    assert lib.start(s, 0x2000, 0x3000) == 0                     # is to wait for the first call; its launch fails
    assert lib.end(700) == 700
    assert lib.start(s, 0x2000, 0x4000) == 0                     # the first call may still be writing
    assert lib.end(0) == 0
    assert lib.start(s, 0x5000, 0x6000) == 1
