"""The packed square root of the noise generator against CUDA's correctly rounded one, for every argument the generator can
produce: x = -2 ln u for all 2^24 values of u, and the two halves of the packed operation with different arguments."""
import ctypes as C
import os
import subprocess

import pytest
import torch

from paper_2202_05008_b200 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "noise.cuh"
using namespace evo;
__global__ void check(unsigned long long* wrong)
{
    const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x + 1u, other = (k * 2654435761u >> 8) + 1u;    // 1 .. 2^24
    const fp2 x = fp2_mul(fp2_both(-2.0f), ln_of_u24(k, other));
    float a, b, ra, rb;
    fp2_split(x, a, b);
    fp2_split(sqrt_rn2(x), ra, rb);
    if (__float_as_uint(ra) != __float_as_uint(__fsqrt_rn(a)) || __float_as_uint(rb) != __float_as_uint(__fsqrt_rn(b))) atomicAdd(wrong, 1ull);
}
extern "C" int run(unsigned long long* wrong) { check<<<1 << 16, 256>>>(wrong); return cudaDeviceSynchronize(); }
"""


def test_square_roots_of_all_arguments_are_correctly_rounded(tmp_path):
    src, lib = tmp_path / "root.cu", tmp_path / "root.so"
    src.write_text(SOURCE)
    subprocess.check_call([B._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "--shared", "-Xcompiler", "-fPIC",
                           "-I", B.CSRC, "-o", str(lib), str(src)])
    wrong = torch.zeros(1, dtype=torch.int64, device="cuda")
    L = C.CDLL(os.fspath(lib))
    L.run.argtypes = [C.c_void_p]
    assert L.run(wrong.data_ptr()) == 0
    assert int(wrong) == 0
