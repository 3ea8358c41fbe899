"""consumers_stop of stream.cuh, in a kernel of its own: whichever consumer's wait
ran out (lane 0 of a warp or another, any warp), every consumer leaves and the
error is raised; without one, they leave after the last item only and no error
is raised. Nothing here waits."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

THREADS = 128
SOURCE = """
#include "stream.cuh"
__global__ void stop_kernel(int dead, int last, unsigned* err, int* left) {
    left[threadIdx.x] = eiger::consumers_stop<%d>((int)threadIdx.x == dead, last != 0, err);
}
extern "C" int run(int dead, int last, unsigned* err, int* left) {
    stop_kernel<<<1, %d>>>(dead, last, err, left);
    return (int)cudaDeviceSynchronize();
}
""" % (THREADS, THREADS)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2607_04489_gb300 import build

    tmp = tmp_path_factory.mktemp("stream")
    src, so = tmp / "stop.cu", tmp / "libstop.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, "-I",
                    os.path.join(os.path.dirname(build.HERE), "include"), "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("dead", [-1, 0, 5, 31, 32, 77, THREADS - 1])
@pytest.mark.parametrize("last", [0, 1])
def test_consumers_stop(lib, dead, last):
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    left = torch.full((THREADS,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert lib.run(dead, last, ctypes.c_void_p(err.data_ptr()), ctypes.c_void_p(left.data_ptr())) == 0
    np.testing.assert_array_equal(left.cpu().numpy(), int(dead >= 0 or last))
    assert int(err) == (2 if dead >= 0 else 0)  # kErrInternal
