"""The integer conversions between FP32 and FP64 (internal.cuh) against the conversion instructions, bit for
bit: every FP32 word; and the FP64 values at, just above and just below every FP32 value and every tie
between two of them, with random FP64 words of all exponents."""
import ctypes as C
import os
import subprocess

import pytest
import torch

from paper_0912_1976_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "internal.cuh"
using namespace vemg;

// out[0], out[1]: words whose conversions differ; out[2]: an FP64 one of them
__global__ void k_compare(unsigned long long *out) {
    const unsigned step[] = {0u, 1u, 0x0fffffffu, 0x10000000u, 0x10000001u, 0x1fffffffu};
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    for (unsigned long long w = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; w >> 32 == 0; w += stride) {
        const float f = __uint_as_float((unsigned)w);
        const double d = (double)f;
        if (__double_as_longlong(cvt_f64(f)) != __double_as_longlong(d)) atomicAdd(out, 1ull);
        for (int k = 0; k < 7; ++k) {
            // the last: a scrambled word
            unsigned long long u = k < 6 ? (unsigned long long)__double_as_longlong(d) + step[k]
                                         : (w * 0x9e3779b97f4a7c15ull) ^ (w << 31);
            asm volatile("" : "+l"(u));   // or the compiler takes f for (float)(double)f, a signalling NaN included
            const double x = __longlong_as_double((long long)u);
            if (__float_as_uint(cvt_f32(x)) != __float_as_uint(__double2float_rn(x))) {
                atomicAdd(out + 1, 1ull);
                out[2] = u;
            }
        }
    }
}

extern "C" int compare(unsigned long long *out, cudaStream_t s) {
    k_compare<<<1216, 256, 0, s>>>(out);
    return (int)cudaGetLastError();
}
"""


def test_conversions_are_those_of_the_instructions(tmp_path):
    src, lib = tmp_path / "convert.cu", tmp_path / "libconvert.so"
    src.write_text(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, *B.COMMON, "-I", B.CSRC, "-shared", str(src), "-o", str(lib), "-lcudart"],
                   check=True)
    out = torch.zeros(3, dtype=torch.int64, device="cuda")
    rc = C.CDLL(os.fspath(lib)).compare(C.c_void_p(out.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0 and out.tolist() == [0, 0, 0], [hex(v & 2 ** 64 - 1) for v in out.tolist()]
