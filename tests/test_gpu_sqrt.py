"""The square roots of the noise against FP64 square roots, on the device.

Heron's step from the hardware reciprocal square root (relative error at most 2^-22.9)
leaves at most 2^-24 (1 + 2^-20) of the result, by the derivation beside sqrt_heron; every
mantissa of both exponent parities, at exponents from 2^-100 to 2^100, one value at a time and
in pairs, with and without the test of the sign.
"""
import ctypes
import subprocess

import pytest

from paper_2006_12910_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_dev.cuh"
using namespace lbmk;
__global__ void k(int ex, double* worst) {
    double w = 0.0;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < (1u << 24); i += gridDim.x * blockDim.x) {
        const float x = __uint_as_float(((uint32_t)(127 + ex) << 23) + i);  // [2^ex, 2^(ex + 2))
        const double s = sqrt((double)x);
        const float y = rsqrt_hw(x);
        const float2 p = sqrt_heron(make_float2(x, 1.0f)), n = neg_sqrt(make_float2(-1.0f, -x), make_float2(1.0f, y));
        w = fmax(w, fabs(sqrt_heron(x) / s - 1.0));
        w = fmax(w, fabs(p.x / s - 1.0));
        w = fmax(w, fabs(-neg_sqrt(-x, y) / s - 1.0));
        w = fmax(w, fabs(-n.y / s - 1.0));
        w = fmax(w, fabs(p.y - 1.0) + fabs(n.x + 1.0));
    }
    atomicMax((unsigned long long*)worst, (unsigned long long)__double_as_longlong(w));
}
__global__ void z(float* out) {
    out[0] = sqrt_heron(0.0f);
    out[1] = sqrt_heron(-1.0f);
}
extern "C" int worst(int ex, double* out) {
    double* d;
    if (cudaMalloc(&d, 8) != cudaSuccess || cudaMemset(d, 0, 8) != cudaSuccess) return 1;
    k<<<1216, 256>>>(ex, d);
    const int r = cudaMemcpy(out, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(d);
    return r;
}
extern "C" int zeros(float* out) {
    float* d;
    if (cudaMalloc(&d, 8) != cudaSuccess) return 1;
    z<<<1, 1>>>(d);
    const int r = cudaMemcpy(out, d, 8, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(d);
    return r;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    d = tmp_path_factory.mktemp("sqrt")
    (d / "s.cu").write_text(SOURCE)
    subprocess.run([build._nvcc(), "-shared", str(d / "s.cu"), "-o", str(d / "s.so")] + build._flags(), check=True,
                   capture_output=True)
    return ctypes.CDLL(str(d / "s.so"))


@pytest.mark.parametrize("ex", [-100, -51, -24, -22, -2, 0, 2, 4, 5, 98])
def test_square_root(lib, ex):
    out = ctypes.c_double(0.0)
    assert lib.worst(ex, ctypes.byref(out)) == 0
    assert 0.0 < out.value <= 2.0 ** -24 * (1 + 2.0 ** -20), out.value * 2 ** 24


def test_no_square_root_of_what_is_not_positive(lib):
    out = (ctypes.c_float * 2)(1.0, 1.0)
    assert lib.zeros(out) == 0
    assert list(out) == [0.0, 0.0]
