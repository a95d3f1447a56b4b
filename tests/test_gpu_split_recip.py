"""The split path's FP32 reciprocal and square root (csrc/dg_cell.cuh) are the correctly rounded ones: all 2^23
mantissas, at exponents over the range (even and odd ones for the root)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MAIN = r"""
#include "dg_line.cuh"
#include <cstdio>
using namespace crkdg;
__global__ void compare(int e, unsigned long long *differ) {
    const float x = __uint_as_float(((unsigned)(e + 127) << 23) | (blockIdx.x * 256u + threadIdx.x));
    if (__float_as_uint(pc::recip_f(x)) != __float_as_uint(__frcp_rn(x))) atomicAdd(differ, 1ull);
    if (__float_as_uint(pc::root_f(x)) != __float_as_uint(__fsqrt_rn(x))) atomicAdd(differ + 1, 1ull);
}
int main() {
    unsigned long long *d, h[2];
    if (cudaMalloc(&d, sizeof(h)) != cudaSuccess || cudaMemset(d, 0, sizeof(h)) != cudaSuccess) return 2;
    const int exponents[] = {-126, -98, -60, -47, -13, -1, 0, 1, 2, 17, 60, 101, 125};
    for (int e : exponents) compare<<<(1 << 23) / 256, 256>>>(e, d);
    if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    printf("%llu %llu\n", h[0], h[1]);
    return 0;
}
"""


def test_correctly_rounded(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_16002_gb300.build import ARCH, CSRC, FLAGS, _nvcc

    (tmp_path / "main.cu").write_text(MAIN)
    exe = str(tmp_path / "main")
    r = subprocess.run([_nvcc(), *ARCH, *FLAGS, "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(tmp_path / "main.cu"),
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.split() == ["0", "0"]
