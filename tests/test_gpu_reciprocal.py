"""The FP32 transport's reciprocal and square root against CUDA's correctly rounded
functions, for every float of the range they are used on."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include <cstdio>
#include "spmc_transport_f32.cuh"
// bit patterns [lo, hi]: counts of values that differ from __frcp_rn and __fsqrt_rn
__global__ void compare(unsigned lo, unsigned hi, unsigned long long *bad) {
    unsigned long long r = 0, s = 0;
    for (unsigned long long i = lo + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i <= hi;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((unsigned)i);
        r += __float_as_uint(spmc::rcp_normal(x)) != __float_as_uint(__frcp_rn(x));
        s += __float_as_uint(spmc::sqrt_normal(x)) != __float_as_uint(__fsqrt_rn(x));
    }
    if (r) atomicAdd(bad, r);
    if (s) atomicAdd(bad + 1, s);
}
int main() {
    unsigned long long *d = nullptr, h[2] = {1, 1};
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
    compare<<<608, 256>>>((127u - 100u) << 23, (127u + 100u) << 23, d);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%llu %llu\n", h[0], h[1]);
    return 0;
}
"""


@pytest.mark.gpu
def test_every_float_of_the_range(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_13929_gb300 import build
    src, exe = tmp_path / "compare.cu", tmp_path / "compare"
    src.write_text(PROGRAM)
    # without -fmad=false and with -O3, as the kernel itself is built
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", build.ARCH, "--expt-relaxed-constexpr", f"-I{build.CSRC}",
                    f"-I{build.INCLUDE}", "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    assert out.split() == ["0", "0"]


def test_scattering_denominator_stays_in_the_range():
    """1 - g + 2 g u for every g the entry points take, u at the ends of its range, with and
    without a fused product: between 2^-24 and 4."""
    f = np.float32
    g = np.concatenate([np.nextafter([1.0, -1.0], 0.0), 1.0 - 2.0 ** -np.arange(1, 53), 2.0 ** -np.arange(1, 53) - 1.0,
                        np.linspace(-0.999, 0.999, 4001)])
    g = g.astype(f)                               # +-1 among them, as |g| < 1 rounds in FP32
    a, b = f(1.0) - g, f(2.0) * g
    for u in (f(2.0 ** -24), f(0.5), f(1.0 - 2.0 ** -24)):
        plain = a + b * u
        fused = (a.astype(np.float64) + b.astype(np.float64) * np.float64(u)).astype(f)
        for d in (plain, fused):
            assert d.dtype == f and d.min() >= 2.0 ** -24 and d.max() <= 4.0
