"""The traversals' own elementary functions on the GPU (opacity and reciprocals: the emission-absorption reading of
Sec. 6.2, the pixel ray of Sec. 6.1) against FP64 or exact references, at the bounds their comments state. The functions are
device code without an entry point, so a small library around their headers is compiled here."""
import ctypes
import os
import subprocess
from fractions import Fraction as Q

import numpy as np
import pytest

from paper_1704_02724_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "canvox_internal.cuh"
#include "opacity.cuh"
using namespace canvox;
__device__ void most(double e, unsigned long long* w) { atomicMax(w, (unsigned long long)__double_as_longlong(e)); }
__device__ double ulps32(double got, double want) {  // in units of the binary32 spacing at `want`
    const int e = (int)((__double_as_longlong(fabs(want)) >> 52) & 0x7FF) - 1023;
    return fabs(got - want) / ldexp(1.0, max(e, -126) - 23);
}
// every binary32 value with the patterns [lo, hi)
__global__ void all32(unsigned lo, unsigned hi, unsigned long long* w) {
    double worst = 0.0;
    for (unsigned long long u = lo + (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; u < hi;
         u += (unsigned long long)gridDim.x * blockDim.x) {
        const float x = __int_as_float((int)(unsigned)u);
        const double e = ulps32((double)expm1_neg(x), expm1(-(double)x));
        worst = e > worst || e != e ? e : worst;
    }
    most(worst, w);
}
__global__ void rcp(const double* x, int n, unsigned long long* w) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double r = rcp64(x[i]);
    const double ulp = __longlong_as_double((__double_as_longlong(r) & 0x7FF0000000000000ll)) * 2.220446049250313e-16;
    most(fabs(fma(-x[i], r, 1.0)) / (x[i] * ulp), w);  // (the residual is exact)
}
__global__ void op64(const double* x, int n, double* y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = expm1_neg64(x[i]);
}
static double finish(unsigned long long* w) {
    double r = -1.0;
    if (cudaMemcpy(&r, w, 8, cudaMemcpyDeviceToHost) != cudaSuccess) r = -1.0;
    cudaFree(w);
    return r;
}
extern "C" double worst32(unsigned lo, unsigned hi) {
    unsigned long long* w;
    if (cudaMalloc(&w, 8) != cudaSuccess) return -1.0;
    cudaMemset(w, 0, 8);
    all32<<<152 * 8, 256>>>(lo, hi, w);
    return finish(w);
}
extern "C" double worst_rcp(const double* host, int n) {
    unsigned long long* w;
    double* x;
    if (cudaMalloc(&w, 8) != cudaSuccess || cudaMalloc(&x, 8 * (size_t)n) != cudaSuccess) return -1.0;
    cudaMemset(w, 0, 8);
    cudaMemcpy(x, host, 8 * (size_t)n, cudaMemcpyHostToDevice);
    rcp<<<(n + 255) / 256, 256>>>(x, n, w);
    const double r = finish(w);
    cudaFree(x);
    return r;
}
extern "C" int opacity64(const double* host, int n, double* out) {
    double *x, *y;
    if (cudaMalloc(&x, 8 * (size_t)n) != cudaSuccess || cudaMalloc(&y, 8 * (size_t)n) != cudaSuccess) return -1;
    cudaMemcpy(x, host, 8 * (size_t)n, cudaMemcpyHostToDevice);
    op64<<<(n + 255) / 256, 256>>>(x, n, y);
    const int e = (int)cudaMemcpy(out, y, 8 * (size_t)n, cudaMemcpyDeviceToHost);
    cudaFree(x);
    cudaFree(y);
    return e;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("device_math")
    (d / "m.cu").write_text(SOURCE)
    so = str(d / "device_math.so")
    subprocess.run([_build.NVCC] + _build.FLAGS + ["-I", _build.CSRC, "-shared", str(d / "m.cu"), "-o", so], check=True)
    L = ctypes.CDLL(os.path.abspath(so))
    L.worst32.argtypes, L.worst32.restype = [ctypes.c_uint32, ctypes.c_uint32], ctypes.c_double
    L.worst_rcp.argtypes, L.worst_rcp.restype = [ctypes.c_void_p, ctypes.c_int], ctypes.c_double
    L.opacity64.argtypes, L.opacity64.restype = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p], ctypes.c_int
    return L


def _bits(x):
    return int(np.float32(x).view(np.uint32))


@pytest.mark.parametrize("lo,hi", [(2.0 ** -40, 1.0), (1.0, 2.0 ** 27), (-2.0 ** -40, -0.25)])
def test_opacity_within_an_ulp(lib, lo, hi):
    """Every binary32 argument: both sides of 1, up to the longest opaque segments, and the slightly negative ones."""
    assert 0.0 < lib.worst32(_bits(lo), _bits(hi)) <= 1.0


def test_opacity_at_zero(lib):
    assert lib.worst32(_bits(0.0), 1) == 0.0 and lib.worst32(_bits(-0.0), _bits(-0.0) + 1) == 0.0


@pytest.mark.parametrize("span", [1, 60, 1000])
def test_reciprocal(lib, span):
    """Half an ulp, and e^3 <= 2^-58 of an approximation of 19.5 bits or more."""
    rng = np.random.default_rng(span)
    x = np.ldexp(1.0 + rng.random(1 << 22), -rng.integers(1, span + 1, 1 << 22))
    x[:4] = 1.0, 0.5, np.nextafter(1.0, 0.0), np.nextafter(0.5, 1.0)
    assert 0.0 < lib.worst_rcp(x.ctypes.data, len(x)) <= 0.5 + 2.0 ** -5


def test_fp64_opacity(lib):
    """On both sides of the switch at 1/8 and down to 2^-60, against the exact series (to 2^-90)."""
    rng = np.random.default_rng(8)
    x = np.concatenate([np.exp(rng.uniform(np.log(2.0 ** -60), np.log(0.125), 3000)), rng.uniform(0.12, 0.13, 1000),
                        rng.uniform(0.125, 4.0, 500), [0.125, np.nextafter(0.125, 0.0), -1e-12, -1e-3]])
    got = np.zeros_like(x)
    assert lib.opacity64(x.ctypes.data, len(x), got.ctypes.data) == 0
    for v, g in zip(x, got):
        y, term, want, k = -Q(float(v)), Q(1), Q(0), 0
        while k < 2 or abs(term) > abs(want) / 2 ** 90:
            k += 1
            term = Q((term * y / k * 2 ** 300).__round__(), 2 ** 300)   # (kept to 2^-300: exact fractions grow)
            want += term
        assert abs(Q(float(g)) - want) <= abs(want) / 2 ** 52, v
