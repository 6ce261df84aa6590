"""Dynamic shared-memory limits (csrc/smem.cu) against a fake of the CUDA call:
each kernel's limit is set once per larger size and never lowered, however many
kernels a process uses and from however many threads."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1509_04685_gb300", "csrc")

FAKE = r"""
#include <cuda_runtime_api.h>
#include <map>
#include <mutex>
#include <thread>
#include <vector>
#include "smem.h"
namespace cola { int g_last_cuda_error = 0; }
static std::mutex m;
static std::map<const void*, int> limit;
static int calls = 0, lowered = 0, refuse = 0;
extern "C" {
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    std::lock_guard<std::mutex> g(m);
    if (refuse) return cudaErrorInvalidValue;
    ++calls;
    if (limit.count(f) && v < limit[f]) ++lowered;
    limit[f] = v;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
int t_set(long fn, long bytes) { return cola::set_smem((const void*)fn, (size_t)bytes); }
void t_refuse(int on) { refuse = on; }
int t_error(void) { return cola::g_last_cuda_error; }
int t_calls(void) { return calls; }
int t_lowered(void) { return lowered; }
int t_limit(long fn) { return limit.count((const void*)fn) ? limit[(const void*)fn] : 0; }
// threads that each ask for growing sizes of the same kernels
void t_threads(int n, long first, int kernels) {
    std::vector<std::thread> t;
    for (int i = 0; i < n; ++i)
        t.emplace_back([=] {
            for (int b = 50; b <= 200; b += 10)
                for (int k = 0; k < kernels; ++k) cola::set_smem((const void*)(first + k), (size_t)b * 1024);
        });
    for (auto& x : t) x.join();
}
}
"""


@pytest.fixture()
def smem(tmp_path):
    from paper_1509_04685_gb300.build import nvcc
    inc = os.path.join(os.path.dirname(os.path.dirname(nvcc())), "include")
    src, lib = tmp_path / "fake.cpp", tmp_path / "libfake.so"
    src.write_text(FAKE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic", "-I", inc, "-I", CSRC, "-x", "c++",
                    os.path.join(CSRC, "smem.cu"), str(src), "-o", str(lib)], check=True)
    lib = ctypes.CDLL(str(lib))
    lib.t_set.argtypes = [ctypes.c_long, ctypes.c_long]
    lib.t_limit.argtypes = [ctypes.c_long]
    lib.t_threads.argtypes = [ctypes.c_int, ctypes.c_long, ctypes.c_int]
    return lib


def test_no_kernel_is_set_twice_however_many_there_are(smem):
    for k in range(1, 201):
        assert smem.t_set(k, 100 * 1024)
    assert smem.t_calls() == 200
    for k in range(1, 201):  # what a stream capture would do: nothing left to set
        assert smem.t_set(k, 100 * 1024) and smem.t_set(k, 50 * 1024)
    assert smem.t_calls() == 200


def test_a_limit_is_raised_and_never_lowered(smem):
    for k in range(1, 201):
        for kb in (60, 200, 90, 150):  # a runtime kernel's size goes with the mesh
            assert smem.t_set(k, kb * 1024)
        assert smem.t_limit(k) == 200 * 1024
    assert smem.t_lowered() == 0
    assert smem.t_set(999, 40 * 1024) and smem.t_limit(999) == 0  # fits without


def test_threads_take_turns(smem):
    smem.t_threads(8, 1, 100)
    assert smem.t_lowered() == 0
    assert all(smem.t_limit(k) == 200 * 1024 for k in range(1, 101))
    assert smem.t_calls() == 16 * 100  # one call per kernel and size


def test_a_refusal_is_reported_and_not_remembered(smem):
    smem.t_refuse(1)
    assert not smem.t_set(7, 100 * 1024)
    assert smem.t_error() != 0
    smem.t_refuse(0)
    assert smem.t_set(7, 100 * 1024) and smem.t_limit(7) == 100 * 1024
