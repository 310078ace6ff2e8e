"""A build whose gather fails between the fork and the join of its two streams
waits for the side stream before it gives buffers back.  The host code is run
against a fake CUDA runtime that logs its calls and fails the chosen one."""
import os
import subprocess

import pytest

from paper_1906_12018_gb300 import build_ext

FAKE = r"""
#include <cstdlib>
#include "plb_host.cuh"

extern int left;

namespace plb {
__global__ void k_gp_warp(GpParams) {}
__global__ void k_gp_block(GpParams) {}
cudaError_t dev_alloc(void** p, size_t bytes, cudaStream_t) { *p = std::malloc(bytes); return cudaSuccess; }
}  // namespace plb

int main(int, char** argv) {
    const cudaStream_t s = (cudaStream_t)1;
    plb::DevPool pool(s);
    plb::RoundCounters ctr{};
    pool.alloc<int>(4);
    plb::SideStream side;
    if (side.create() != cudaSuccess) return 2;
    left = std::atoi(argv[1]);
    const cudaError_t e = plb::launch_tiers(plb::GpParams{}, plb::GpParams{}, plb::SplitLists{}, nullptr, nullptr, &ctr,
                                            1, 0, 1, 64, 0, s, side, nullptr);
    std::printf(e == cudaSuccess ? "ok " : "failed ");
    return 0;
}
"""

# the runtime's calls, and those of nvcc's launch code
STUBS = r"""
#include <cstdio>
#include <cuda_runtime_api.h>

int left = 1 << 30;  // calls until the one that fails
static cudaError_t log(const char* what, const void* stream) {
    if (--left == 0) {
        std::printf("%s:fails ", what);
        return cudaErrorUnknown;
    }
    std::printf("%s:%ld ", what, (long)(size_t)stream);
    return cudaSuccess;
}

extern "C" {
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)2; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)8; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)9; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t s) { return log("record", s); }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned) { return log("wait", s); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { std::printf("sync:%ld ", (long)(size_t)s); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::printf("destroy:%ld ", (long)(size_t)s); return cudaSuccess; }
cudaError_t cudaFreeAsync(void*, cudaStream_t s) { std::printf("free:%ld ", (long)(size_t)s); return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
char __cudaInitModule(void**) { return 0; }
static cudaStream_t pushed;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t s) { pushed = s; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void* s) { *(cudaStream_t*)s = pushed; return cudaSuccess; }
cudaError_t __cudaGetKernel(void**, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, cudaStream_t s) {
    std::printf("kernel:%ld ", (long)(size_t)s);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t s) {
    return __cudaLaunchKernel(nullptr, dim3(), dim3(), nullptr, 0, s);
}
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("side")
    for name, src in (("fake.cu", FAKE), ("stubs.cpp", STUBS)):
        (d / name).write_text(src)
    exe = str(d / "fake")
    r = subprocess.run([build_ext._nvcc(), *build_ext.ARCH, "-std=c++17", "-I", build_ext.INCLUDE, "-I", build_ext.CSRC,
                        "-cudart", "none", str(d / "fake.cu"), str(d / "stubs.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def calls(program, fails):
    return subprocess.run([program, str(fails)], capture_output=True, text=True, check=True).stdout.split()


def test_a_gather_that_succeeds_does_not_wait(program):
    log = calls(program, 1 << 30)
    assert log == ["record:1", "wait:2", "kernel:2", "kernel:1", "record:2", "wait:1", "kernel:1", "ok", "destroy:2",
                   "free:1"]


@pytest.mark.parametrize("fails", [1, 2, 3, 4])
def test_a_gather_that_fails_waits_for_what_it_launched(program, fails):
    log = calls(program, fails)
    assert "failed" in log and log[-2:] == ["destroy:2", "free:1"]
    assert ("sync:2" in log) == ("kernel:2" in log)
    assert "sync:2" not in log or log.index("kernel:2") < log.index("sync:2") < log.index("free:1")
