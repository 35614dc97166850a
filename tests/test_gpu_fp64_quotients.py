"""div_d of csrc/fp64.cuh where the dividend or the quotient leaves the moderate range: zeros,
infinities, NaN, subnormal numbers, quotients that overflow or underflow.  As CUDA's division
gives them: the same special values, else within a unit in the last place (the last step is one
rounding of a value within 2^-60), below the smallest normal number within one subnormal step."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2601_03935_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cmath>
#include "fp64.cuh"
using namespace gsis;
__device__ unsigned long long g_worst;
__global__ void check(int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * n) return;
    const double special[] = {0.0, 1.0, 3.0, INFINITY, NAN, 5e-324, 1.5e-310, 2.2250738585072014e-308,
                              1.7976931348623157e308, 1e300, 1e-300, 0.1};
    // the special values and powers of two times odd numbers over the whole range, either sign
    auto value = [&](int k) {
        const double x = k < 24 ? special[k / 2] : ldexp(1.0 + (k * 37 % 101) / 128.0, -1070 + (k - 24) * 2);
        return k & 1 ? -x : x;
    };
    const double a = value(i / n), b = value(i % n), q = a / b, d = fp64::div_d(a, b);
    double off = 1e300;
    if (d == q || (isnan(d) && isnan(q))) off = signbit(d) == signbit(q) || isnan(q) ? 0.0 : 1e300;
    else if (isfinite(q) && isfinite(d))
        off = fabs(d - q) / (__longlong_as_double(__double_as_longlong(fabs(q)) + 1) - fabs(q));
    atomicMax(&g_worst, (unsigned long long)__double_as_longlong(off));
}
int main() {
    const int n = 24 + 1046;
    check<<<(n * n + 127) / 128, 128>>>(n);
    double h;
    if (cudaMemcpyFromSymbol(&h, g_worst, sizeof h) != cudaSuccess) return 1;
    printf("%.6g\n", h);
    return 0;
}
"""


@pytest.mark.gpu
def test_quotients_at_the_edges(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "div_check.cu", tmp_path / "div_check"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    worst = float(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout)
    assert worst <= 1.0, worst
