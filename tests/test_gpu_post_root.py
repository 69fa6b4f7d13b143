"""The tiled field's square root of a pair against sqrtf, over every significand at two adjacent
exponents, three times: equal but for a handful of arguments, and there by one ulp."""
import ctypes
import os
import subprocess

import pytest

from paper_2403_11156_gb300 import build

from gpu_util import gpu_ctx  # noqa: F401  (builds the library)

pytestmark = pytest.mark.gpu

SOURCE = """
#include "sph_grid.cu"
#include "sph_post.cu"
namespace sph {
__global__ void k_root(uint32_t first, uint32_t *out)
{
    const uint32_t i = first + blockIdx.x * blockDim.x + threadIdx.x;
    const float a = __uint_as_float(i), b = __uint_as_float(i ^ 1u);
    float ra, rb;
    unpack(sqrt2(pack_xy(a, b), a, b), ra, rb);
    const int da = abs((int)(__float_as_uint(ra) - __float_as_uint(sqrtf(a))));
    const int db = abs((int)(__float_as_uint(rb) - __float_as_uint(sqrtf(b))));
    if (da) atomicAdd(out, 1u);
    atomicMax(out + 1, (uint32_t)max(da, db));
}
}  // namespace sph
extern "C" int roots(uint32_t first, uint32_t *out)
{
    sph::k_root<<<1 << 16, 256>>>(first, out);
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


def test_root_of_pairs(tmp_path):
    import torch
    src = tmp_path / "root.cu"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(tmp_path / "root.so"), str(src)], check=True)
    lib = ctypes.CDLL(os.fspath(tmp_path / "root.so"))
    lib.roots.argtypes = [ctypes.c_uint32, ctypes.c_void_p]
    for exponent in (127 - 60, 127 - 10, 127):       # 2^24 numbers from 2^(exponent - 127) on
        out = torch.zeros(2, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert lib.roots(exponent << 23, out.data_ptr()) == 0
        differ, ulps = out.tolist()
        assert differ <= 4 and ulps <= 1, (exponent, differ, ulps)
