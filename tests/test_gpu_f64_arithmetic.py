"""The FP64 reciprocal, quotient and square roots written out for this library, over 2^28 arguments of every exponent
that the kernels meet (2^-300 .. 2^300) and densely around the densities' 1, in units of the result's last place.

Bounds, from the starting approximations' relative error e (checked first: at most 2^-19, two roundings to 20
fraction bits): the reciprocal's third-order step leaves e^3 <= 2^-57, a sixteenth of a unit at most, beside the
last rounding's half; a quotient and a square root end in a correction by their exact residual, which leaves the
last rounding.  Their special values: the square root of 0 and of subnormal numbers is 0, of a negative number
NaN."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1310_7450_gb300", "csrc")
SOURCE = r"""
#include <cstdio>
#include "lb_warmstart.cu"
using namespace lbk;
__device__ unsigned long long mix(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
// a positive number: random fraction bits, exponent in [-300, 300] (near: in [1/2, 2))
__device__ double number(unsigned long long k, bool near) {
    const unsigned long long a = mix(2 * k * 0x9E3779B97F4A7C15ull + 1), b = mix((2 * k + 1) * 0x9E3779B97F4A7C15ull);
    const int e = near ? (int)(b & 1) - 1 : (int)(b % 601) - 300;
    return __longlong_as_double((long long)((a >> 12) | ((unsigned long long)(1023 + e) << 52)));
}
__device__ double ulp(double x) { return __longlong_as_double((__double_as_longlong(x) & 0x7ff0000000000000ll) - (52ll << 52)); }
__device__ void worst(double* out, double v) {  // v >= 0, or NaN (orders above every number)
    atomicMax((long long*)out, __double_as_longlong(fabs(v)));
}
__global__ void k_errors(double* out) {  // out[0..1] starting errors, [2] reciprocal, [3] quotient, [4] root, [5] root (warm start)
    double m[6] = {};
    for (unsigned long long k = blockIdx.x * blockDim.x + threadIdx.x; k < (1ull << 28); k += gridDim.x * blockDim.x) {
        const bool near = k & 1;
        const double x = number(k, near), a = number(k ^ 0x5555555555ull, near);
        double y, r;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
        m[0] = fmax(m[0], fabs(__fma_rn(-x, y, 1.0)));
        m[1] = fmax(m[1], 0.5 * fabs(__fma_rn(-x * r, r, 1.0)));
        const double c = Arith<double>::rcp(x), q = Arith<double>::div(a, x), g = Arith<double>::sqrt(x), w = ws_sqrt(x);
        const double e[4] = {__fma_rn(-x, c, 1.0) / x / ulp(c), __fma_rn(-x, q, a) / x / ulp(q),
                             __fma_rn(-g, g, x) / (g + g) / ulp(g), __fma_rn(-w, w, x) / (w + w) / ulp(w)};
        for (int j = 0; j < 4; ++j) m[2 + j] = e[j] == e[j] ? fmax(m[2 + j], fabs(e[j])) : 1e300;
    }
    for (int j = 0; j < 6; ++j) worst(out + j, m[j]);
}
__global__ void k_special(double* out) {
    out[0] = Arith<double>::sqrt(0.0);
    out[1] = Arith<double>::sqrt(4e-320);
    out[2] = Arith<double>::sqrt(-1.0);
    out[3] = Arith<double>::div(0.0, 3.0);
}
int main() {
    double *d, h[10];
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
    k_errors<<<608, 256>>>(d);
    k_special<<<1, 1>>>(d + 6);
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    for (double v : h) std::printf("%.17g\n", v);
}
"""


@pytest.fixture(scope="module")
def measured(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("f64")
    (d / "f64.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), str(d / "f64.cu"), "-o", str(d / "f64")], check=True)
    out = subprocess.run([str(d / "f64")], check=True, capture_output=True, text=True).stdout
    return [float(x) for x in out.split()]


def test_errors_in_units_of_the_last_place(measured):
    rcp0, rsqrt0, rcp, div, root, ws_root = measured[:6]
    print(f"start: 1/x {rcp0:.3e}, 1/sqrt(x) {rsqrt0:.3e}; units: 1/x {rcp:.5f}, a/x {div:.5f}, sqrt {root:.5f}, warm start {ws_root:.5f}")
    assert rcp0 <= 2.0 ** -19 and rsqrt0 <= 2.0 ** -19
    assert rcp <= 0.5 + 0.0625 + 0.001
    assert div <= 0.501 and root <= 0.501 and ws_root <= 0.501


def test_special_values(measured):
    zero, subnormal, negative, quotient = measured[6:]
    assert zero == 0.0 and subnormal == 0.0 and negative != negative and quotient == 0.0
