"""The descent bounds' packed square root against the device's correctly
rounded one, on every value of its range (marked gpu)."""
import os
import subprocess

import pytest

from paper_1911_10217_gb300 import build

pytestmark = pytest.mark.gpu

# a pair of neighbouring values a turn, from 2^-100 to 2^60, and zero
SOURCE = r"""
#include <cstdio>
#include "rll_device.cuh"
__global__ void compare(uint32_t first, uint32_t count, unsigned long long* tally)
{
    unsigned long long seen = 0, differ = 0;
    const uint32_t stride = gridDim.x * blockDim.x;
    for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; 2 * i < count; i += stride) {
        const float x = __uint_as_float(first + 2 * (uint32_t)i), y = __uint_as_float(first + 2 * (uint32_t)i + 1);
        const float2 r = rll::neg_sqrt2(make_float2(-x, -y));
        seen += 2;
        differ += (-r.x != __fsqrt_rn(x)) + (-r.y != __fsqrt_rn(y));
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const float2 z = rll::neg_sqrt2(make_float2(0.0f, -0.0f));
        seen += 2;
        differ += (z.x != 0.0f) + (z.y != 0.0f);
    }
    atomicAdd(tally, seen);
    atomicAdd(tally + 1, differ);
}
int main()
{
    unsigned long long *d, h[2] = {0, 1};
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
    compare<<<1216, 256>>>(0x0D800000u, 0x50000000u, d);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu\n", h[0], h[1]);
    return 0;
}
"""


def test_packed_square_root_on_every_value(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, exe = tmp_path / "compare.cu", tmp_path / "compare"
    src.write_text(SOURCE)
    subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-I" + build.CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True, cwd=os.path.dirname(build.CSRC))
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    assert out == [str(0x50000000 + 2), "0"]
