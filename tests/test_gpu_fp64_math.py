"""The FP64 functions of csrc/fp64.cuh against CUDA's own over their ranges and at the edges
where they hand over to it: a small program built from the header prints the largest error
of each in units in the last place.

Bounds: an ulp for the reciprocal, quotient and square root (their last step is one
correctly rounded operation on a value within 2^-60); 2 for exp2n (rounded table entry,
rounded result, polynomial within 2^-54); for log the error is 1.5 ulp of max(1, |log x|)
(the sum of a rounded table entry and a rounded tail); for x^p the same times |p| plus the
exponential's 2; the conversions are exact."""
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
__device__ unsigned long long g_max[10];
__device__ void note(int k, double ulps) { atomicMax(&g_max[k], (unsigned long long)__double_as_longlong(ulps)); }
__device__ double ulp(double x) { return __longlong_as_double(__double_as_longlong(fabs(x)) + 1) - fabs(x); }
__device__ double off(double a, double b) {
    if (a == b || (isnan(a) && isnan(b))) return 0.0;
    return isfinite(a) && isfinite(b) ? fabs(a - b) / ulp(b) : 1e300;
}
__global__ void check(int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    unsigned long long s = 0x9E3779B97F4A7C15ull * (i + 1);
    s ^= s >> 30; s *= 0xBF58476D1CE4E5B9ull; s ^= s >> 27; s *= 0x94D049BB133111EBull; s ^= s >> 31;
    const double u = (double)(s >> 11) / 9007199254740992.0;
    const double edge[] = {0.0, -0.0, 1.0, -1.0, INFINITY, -INFINITY, NAN, 5e-324, 2.2250738585072014e-308,
                           1.7976931348623157e308, 1e-300, 1e300, 0.99999999999999989, 1.0000000000000002, 2.0, 0.5};
    const bool at_edge = i < 16;
    // reciprocal, quotient and square root: 2^-300 .. 2^300 and the edges
    const double x = at_edge ? edge[i] : ldexp(1.0 + u, (int)(i % 601) - 300);
    note(0, off(fp64::rcp_d(x), 1.0 / x));
    note(1, off(fp64::div_d(u + 0.25, x), (u + 0.25) / x));
    note(2, off(fp64::sqrt_d(x), sqrt(x)));
    // exp: -760 .. 720 and the edges
    const double y = at_edge ? edge[i] : -760.0 + 1480.0 * ((i % 100000) + u) / 100000.0;
    const double e = exp(y), d = fp64::exp_d(y);
    // the scaled argument carries the rounding of the constant: |y| 2^-53
    note(3, e > 1e-290 && isfinite(e) ? fabs(d - e) / ulp(e) / (1.0 + fabs(y)) : (fabs(d - e) <= 1e-290 || d == e || (isnan(d) && isnan(e)) || y > 709.0 ? 0.0 : 1e300));
    const double l = log(x), ld = fp64::log_d(x);
    note(4, isfinite(l) ? fabs(ld - l) / (2.220446049250313e-16 * fmax(1.0, fabs(l))) : off(ld, l));
    const double t = at_edge ? edge[i] : exp(-7.0 + 14.0 * u), p = -0.5 + (i % 7) * 0.37;
    const double pw = pow(t, p), pd = fp64::pow_d(t, p);
    note(5, at_edge ? (off(pd, pw) > 8.0 ? 1e300 : 0.0) : off(pd, pw) / (4.0 + 2.0 * fabs(p) * fabs(log(t))));
    // conversions: any bit pattern
    const float f = at_edge ? (float)edge[i] : __uint_as_float((unsigned)(s >> 32));
    note(6, off(fp64::widen(f), (double)f));
    const double w = at_edge ? edge[i] : (i & 1) ? __longlong_as_double((long long)s) : ldexp(1.0 + u, (int)(s % 320) - 160) * ((s >> 60) & 1 ? -1 : 1);
    const float a = fp64::narrow(w), b = (float)w;
    note(7, __float_as_uint(a) == __float_as_uint(b) || (isnan(a) && isnan(b)) ? 0.0 : 1.0);
    const double tie = (double)f + ulp((double)f) * 0.0;   // exact floats and midpoints of their neighbours
    const double nx = (double)__uint_as_float(__float_as_uint(f) + 1);
    const float ta = fp64::narrow(0.5 * (tie + nx)), tb = (float)(0.5 * (tie + nx));
    note(7, __float_as_uint(ta) == __float_as_uint(tb) || (isnan(ta) && isnan(tb)) ? 0.0 : 1.0);
    const double q = (u - 0.5) * 4.0;
    note(8, max_pos(fabs(w), q) == fmax(fabs(w), q) || isnan(w) ? 0.0 : 1.0);
    note(8, min_neg(-fabs(w), q) == fmin(-fabs(w), q) || isnan(w) ? 0.0 : 1.0);
    note(9, is_zero(x) == (x == 0.0) && (isnan(x) || x == 0.0 || is_neg(x) == (x < 0.0)) ? 0.0 : 1.0);
}
int main() {
    check<<<(1 << 21) / 128, 128>>>(1 << 21);
    double h[10];
    if (cudaMemcpyFromSymbol(h, g_max, sizeof h) != cudaSuccess) return 1;
    for (int k = 0; k < 10; ++k) printf("%.6g\n", h[k]);
    return 0;
}
"""


@pytest.mark.gpu
def test_errors_against_cuda_functions(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "fp64_check.cu", tmp_path / "fp64_check"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = [float(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    names = ("rcp", "div", "sqrt", "exp", "log", "pow", "widen", "narrow", "max/min", "signs")
    bounds = (1.0, 1.0, 1.0, 2.0, 1.5, 1.0, 0.0, 0.0, 0.0, 0.0)
    assert len(out) == len(names)
    for name, got, bound in zip(names, out, bounds):
        assert got <= bound, "%s: %g > %g" % (name, got, bound)
