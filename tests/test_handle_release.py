"""The order of the runtime's calls when device memory is given back, compiled for the host
against stand-ins of the CUDA runtime.  Handles (csrc/handle.h), one of device 1 dropped while
device 0 is current: the buffers may go only after device 1 was waited for and while it is
current, and not at all when the wait fails.  Buffers (DevBuf, csrc/internal.h): one that grows,
and the others of a call whose allocation is refused, go only after a wait."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1807_08848_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SOURCE = r"""
#include "handle.h"
#include <cstdio>
#include <cstdlib>

static int current = 0;
static cudaError_t sync_result = cudaSuccess, set_result = cudaSuccess;

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) {
    if (set_result != cudaSuccess) return set_result;
    current = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { std::printf("sync %d\n", current); return sync_result; }
cudaError_t cudaGetLastError() { std::printf("clear\n"); return cudaSuccess; }
}

struct Handle {
    ~Handle() { std::printf("free %d\n", current); }
};

int main(int, char** argv) {
    current = std::atoi(argv[1]);
    sync_result = (cudaError_t)std::atoi(argv[2]);
    set_result = (cudaError_t)std::atoi(argv[3]);
    Handle* h = new Handle();
    const cudaError_t e = msp::release_handle(h, 1);
    std::printf("status %d current %d\n", (int)e, current);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime_api.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("handle")
    src, exe = str(d / "main.cpp"), str(d / "main")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", os.path.join(CUDA, "include"), src, "-o", exe], check=True)
    return exe


def run(program, current, sync=0, set_=0):
    r = subprocess.run([program, str(current), str(sync), str(set_)], capture_output=True, text=True, check=True)
    return r.stdout.split("\n")[:-1]


def test_other_device_current(program):
    assert run(program, 0) == ["sync 1", "free 1", "status 0 current 0"]


def test_own_device_current(program):
    assert run(program, 1) == ["sync 1", "free 1", "status 0 current 1"]


def test_failed_wait_keeps_the_memory(program):
    assert run(program, 0, sync=900) == ["sync 1", "clear", "status 900 current 0"]


def test_unusable_device_keeps_the_memory(program):
    assert run(program, 0, set_=101) == ["clear", "status 101 current 0"]


BUFFERS = r"""
#include "internal.h"
#include <cstdio>
#include <cstring>

static bool refuse = false;

extern "C" {
cudaError_t cudaDeviceSynchronize() { std::printf("sync\n"); return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaFree(void*) { std::printf("free\n"); return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
}
namespace msp {
void set_error(const std::string&) {}
msp_status cuda_fail(cudaError_t, const char*, const char*, int) { return MSP_ERR_CUDA; }
cudaError_t pool_alloc(void** p, size_t, cudaStream_t) {
    if (refuse) return cudaErrorMemoryAllocation;
    std::printf("alloc\n");
    *p = (void*)8;
    return cudaSuccess;
}
}  // namespace msp

static msp_status call() {
    msp::DevBuf<double> a, b;
    MSP_TRY(a.alloc(10, nullptr));
    refuse = true;
    MSP_TRY(b.alloc(10, nullptr));
    return MSP_OK;
}

int main(int, char** argv) {
    if (!std::strcmp(argv[1], "grow")) {
        msp::DevBuf<double> a;
        a.alloc(10, nullptr);
        a.alloc(20, nullptr);
        std::printf("end\n");
    } else {
        std::printf("status %d\n", (int)call());
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def buffers(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("buffers")
    src, exe = str(d / "main.cpp"), str(d / "main")
    with open(src, "w") as f:
        f.write(BUFFERS)
    subprocess.run([cxx, "-std=c++17", "-w", "-O1", "-I", CSRC, "-I", os.path.join(CUDA, "include"), src, "-o", exe],
                   check=True)
    return exe


def lines(exe, arg):
    return subprocess.run([exe, arg], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]


def test_growing_buffer_waits(buffers):
    assert lines(buffers, "grow") == ["alloc", "sync", "free", "alloc", "end", "free"]


def test_refused_allocation_waits(buffers):
    assert lines(buffers, "refuse") == ["alloc", "sync", "free", "status -2"]
