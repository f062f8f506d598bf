"""The bounded wait of the asynchronous kernels on its give-up path: whatever the lanes of a warp see, they return the same.

A kernel of one warp, compiled here against the library's header, waits on a barrier of which one phase is complete and the next one
never will be, with the abort flag already raised, so that a wait that cannot succeed ends after its first polls."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1803_04209_b200 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "async.cuh"
using namespace cutoff;
using namespace cutoff::async;
__global__ void k_wait(const int* parity, int* result, DevState* st) {
    __shared__ __align__(8) unsigned long long barrier;
    __shared__ volatile int abort_flag;
    const uint32_t bar = smem_u32(&barrier);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        abort_flag = 1;
        fence_barrier_init();
        mbar_arrive(bar);                     // phase 0 is complete, phase 1 never
    }
    __syncthreads();
    result[threadIdx.x] = mbar_wait(bar, static_cast<uint32_t>(parity[threadIdx.x]), &abort_flag, st);
}
extern "C" int run(const int* parity, int* result, unsigned* error_flags) {
    int *p = nullptr, *r = nullptr;
    DevState* st = nullptr;
    DevState host{};
    cudaError_t e = cudaMalloc(&p, 128);
    if (e == cudaSuccess) e = cudaMalloc(&r, 128);
    if (e == cudaSuccess) e = cudaMalloc(&st, sizeof(DevState));
    if (e == cudaSuccess) e = cudaMemset(st, 0, sizeof(DevState));
    if (e == cudaSuccess) e = cudaMemcpy(p, parity, 128, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_wait<<<1, 32>>>(p, r, st);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(result, r, 128, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&host, st, sizeof(DevState), cudaMemcpyDeviceToHost);
    *error_flags = host.error_flags;
    cudaFree(p); cudaFree(r); cudaFree(st);
    return e;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    build.build()
    folder = tmp_path_factory.mktemp("waits")
    source, library = folder / "waits.cu", folder / "libwaits.so"
    source.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-I", build.CSRC, "-o", os.fspath(library), os.fspath(source)], check=True)
    call = ctypes.CDLL(os.fspath(library)).run

    def run(parity):
        parity = np.asarray(parity, dtype=np.int32)
        result, flags = np.full(32, -1, dtype=np.int32), ctypes.c_uint(0)
        assert call(parity.ctypes.data_as(ctypes.c_void_p), result.ctypes.data_as(ctypes.c_void_p), ctypes.byref(flags)) == 0
        assert flags.value == 0                                     # the other role that aborted has reported it
        return result
    return run


@pytest.mark.parametrize("incomplete", [[], [0], [31], range(1, 32), range(0, 32, 2), range(32)])
def test_a_warp_leaves_a_wait_with_one_result(run, incomplete):
    parity = np.zeros(32, dtype=np.int32)
    parity[list(incomplete)] = 1
    assert np.array_equal(run(parity), np.full(32, 0 if len(incomplete) else 1))
