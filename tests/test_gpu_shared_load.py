"""ld_shared_if (lat_async.cuh), the predicated shared-memory load of the step kernels:
two loads with the same operands, the same constant to fall back on among them, with
a store and a barrier between them give what the memory holds each time. A small
kernel is compiled around the header for it: a block of 64 threads reads its
neighbour's word, every word is rewritten, and the same word is read again."""
import ctypes as C
import os
import subprocess

import pytest
import torch

from paper_0911_5692_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r'''
#include "lat_async.cuh"

template <typename T>
__global__ void twice(T* out)
{
    __shared__ T s[64];
    const int i = threadIdx.x, j = (i + 1) % 64;
    const bool p = i % 3 != 0;
    s[i] = T(i);
    __syncthreads();
    const T a = lat::ld_shared_if(p, s + j, T(0));
    __syncthreads();
    s[i] = T(100 + i);
    __syncthreads();
    const T b = lat::ld_shared_if(p, s + j, T(0));
    out[2 * i] = a;
    out[2 * i + 1] = b;
}

extern "C" int run(void* f, void* d)
{
    twice<float><<<1, 64>>>((float*)f);
    twice<double><<<1, 64>>>((double*)d);
    return (int)cudaDeviceSynchronize();
}
'''


def test_a_second_load_sees_what_was_stored_between(tmp_path):
    src, lib = tmp_path / "twice.cu", tmp_path / "libtwice.so"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                    "-o", str(lib), str(src)], check=True, capture_output=True)
    out = [torch.full((64, 2), -1, dtype=t, device="cuda") for t in (torch.float32, torch.float64)]
    torch.cuda.synchronize()
    assert C.CDLL(str(lib)).run(*[C.c_void_p(o.data_ptr()) for o in out]) == 0
    i = torch.arange(64)
    first = torch.where(i % 3 != 0, (i + 1) % 64, 0)
    second = torch.where(i % 3 != 0, 100 + (i + 1) % 64, 0)
    for o in out:
        assert torch.equal(o.cpu().long(), torch.stack([first, second], dim=1))
