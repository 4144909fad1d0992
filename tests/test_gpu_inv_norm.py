"""inv_norm2, the branch-free 1 / max(1, sqrt(s)) of the unrolled solver's projection, against
sqrtf and the division, bit for bit."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "inv_norm.cuh"
using namespace cslsm;
__global__ void check_kernel(const float *s, size_t n, unsigned *bad, float *first)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n / 2;
         i += (size_t)gridDim.x * blockDim.x) {
        const float2 v = make_float2(s[2 * i], s[2 * i + 1]);
        const float2 r = inv_norm2(v);
        const float ex = 1.f / fmaxf(1.f, sqrtf(v.x)), ey = 1.f / fmaxf(1.f, sqrtf(v.y));
        if (__float_as_uint(r.x) != __float_as_uint(ex) && !atomicAdd(bad, 1u)) *first = v.x;
        if (__float_as_uint(r.y) != __float_as_uint(ey) && !atomicAdd(bad, 1u)) *first = v.y;
    }
}
extern "C" int check(const float *s, size_t n, unsigned *bad, float *first)
{
    check_kernel<<<1024, 256>>>(s, n, bad, first);
    return (int)cudaDeviceSynchronize();
}
"""


def _values():
    man = np.arange(1 << 23, dtype=np.uint32)
    for e in (127, 128):  # every mantissa of an even and an odd exponent
        yield np.uint32(e << 23) | man
    sample = man[:: 4099]
    edges = np.array([0, 1, 2, (1 << 22) - 1, 1 << 22, (1 << 23) - 2, (1 << 23) - 1], np.uint32)
    for e in range(0, 255):  # below 1, and up to the largest exponent
        yield np.uint32(e << 23) | np.concatenate([sample, edges])
    # zero, infinity, NaN
    yield np.array([0, 0x80000000, 0x7F800000, 0x7FC00000], np.uint32)


def test_equals_sqrtf_and_division(tmp_path):
    import torch

    from paper_2511_03093_gb300 import build as b

    src, lib = tmp_path / "check.cu", tmp_path / "check.so"
    src.write_text(SRC)
    subprocess.run([b._nvcc(), "-shared", str(src), "-o", str(lib), *b.NVCC_FLAGS, *b.ARCH],
                   check=True, capture_output=True)
    fn = ctypes.CDLL(str(lib)).check
    bits = np.concatenate(list(_values()))
    bits = np.concatenate([bits, bits[: len(bits) % 2]])
    s = torch.from_numpy(bits.view(np.float32)).cuda()
    bad = torch.zeros(1, dtype=torch.int32, device="cuda")
    first = torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    st = fn(ctypes.c_void_p(s.data_ptr()), ctypes.c_size_t(s.numel()),
            ctypes.c_void_p(bad.data_ptr()), ctypes.c_void_p(first.data_ptr()))
    assert st == 0
    assert int(bad) == 0, (int(bad), float(first))
