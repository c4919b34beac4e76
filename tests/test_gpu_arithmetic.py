"""The arithmetic helpers of the pair sums (needs a GB300): in the FP64 build the reciprocal and the
harmonic mean of two viscosities are correctly rounded, at the ends of the range as well; in single
precision the reciprocal is within 1 ulp and the root within 2.5 for normal results."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2003_01061_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = """
#include "sph_device.cuh"
template <typename T> __global__ void k(int n, const T* a, const T* b, T* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = sph::fast_rcp(a[i]);
    out[n + i] = sph::root_of(a[i]);
    out[2 * n + i] = sph::harmonic<T>(a[i], b[i]);
}
template <typename T> int run(int n, const T* a, const T* b, T* out) {
    T* d = nullptr;
    if (cudaMalloc(&d, 5 * sizeof(T) * n) != cudaSuccess) return 1;
    cudaMemcpy(d, a, sizeof(T) * n, cudaMemcpyHostToDevice);
    cudaMemcpy(d + n, b, sizeof(T) * n, cudaMemcpyHostToDevice);
    k<T><<<(n + 127) / 128, 128>>>(n, d, d + n, d + 2 * n);
    const int bad = cudaMemcpy(out, d + 2 * n, 3 * sizeof(T) * n, cudaMemcpyDeviceToHost) != cudaSuccess;
    cudaFree(d);
    return bad;
}
extern "C" __attribute__((visibility("default"))) int run32(int n, const float* a, const float* b, float* out) { return run<float>(n, a, b, out); }
extern "C" __attribute__((visibility("default"))) int run64(int n, const double* a, const double* b, double* out) { return run<double>(n, a, b, out); }
"""


@pytest.fixture(scope="module")
def arith(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    (d / "arith.cu").write_text(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", "-o", str(d / "arith.so"), str(d / "arith.cu")],
                   check=True)
    lib = C.CDLL(str(d / "arith.so"))

    def go(a, b):
        out = np.empty((3, len(a)), a.dtype)
        run = lib.run64 if a.dtype == np.float64 else lib.run32
        assert run(len(a), a.ctypes.data_as(C.c_void_p), b.ctypes.data_as(C.c_void_p), out.ctypes.data_as(C.c_void_p)) == 0
        return out

    return go


def values(t, n, lo, hi):
    rng = np.random.default_rng(4)
    x = np.exp2(rng.uniform(lo, hi, n))
    x[: n // 2] = 1.0 + rng.random(n // 2)   # one binade, every mantissa alike
    return x.astype(t)


def test_fp64_reciprocal_root_and_harmonic_mean_are_correctly_rounded(arith):
    a, b = values(np.float64, 1 << 21, -300, 300), values(np.float64, 1 << 21, -200, 200)[::-1].copy()
    edge = [0.0, np.inf, np.nan, 5e-324, 2.2e-308, 1.7e308, 1.0, 2.0, np.nextafter(2.0, 0), np.nextafter(1.0, 2)]
    a[: len(edge)], b[: len(edge)] = edge, 0.0
    with np.errstate(all="ignore"):
        rcp, root, s = 1.0 / a, np.sqrt(a), a + b
        harm = np.where(s > 0, 2 * a * b / s, 0.0)
        got = arith(a, b)
    assert np.array_equal(got[0], rcp, equal_nan=True), (got[0] != rcp).sum()
    assert np.array_equal(got[1], root, equal_nan=True)
    assert np.array_equal(got[2], harm, equal_nan=True), (got[2] != harm).sum()


def test_fp32_reciprocal_and_root(arith):
    a, b = values(np.float32, 1 << 21, -100, 100), values(np.float32, 1 << 21, -60, 60)
    got = arith(a, b)
    for g, ref, ulps in ((got[0], 1.0 / a.astype(np.float64), 1.0), (got[1], np.sqrt(a.astype(np.float64)), 2.5)):
        assert (np.abs(g - ref) <= ulps * np.spacing(ref.astype(np.float32))).all()
