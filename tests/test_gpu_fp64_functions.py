"""The FP64 helpers of csrc/mb_fp64.cuh one by one, in a small library compiled
here for the GPU: errors of the reciprocal and the square root from their FMA
residuals and against CUDA's own, over all exponents that their comments
promise, and the promised edges.  Bounds, in units of 2^-53 relative: the
reciprocal's one final rounding (1, its truncation 2^-10 of that), the root's
final rounding and half of one inside (1.5)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "mb_fp64.cuh"
using namespace mbfp;
// out: 16 doubles per input
__global__ void k(const double *x, const double *z, double *out, long long n) {
    const long long t = blockIdx.x * 256LL + threadIdx.x;
    if (t >= n) return;
    const double a = x[t], b = z[t], r = rcp64(a), s = sqrt64(a);
    double *o = out + 16 * t;
    bool ok = true;
    o[0] = r;
    o[1] = __fma_rn(-a, r, 1.0);
    o[2] = __drcp_rn(a);
    o[3] = s;
    o[4] = __fma_rn(-s, s, a);
    o[5] = __dsqrt_rn(a);
    o[6] = pos64(a) ? 1.0 : 0.0;
    o[7] = nonneg64(a) ? 1.0 : 0.0;
    o[8] = min64(a, b);
    o[9] = max64(a, b);
    o[10] = abs64(a);
    o[11] = twice64(a);
    o[12] = half64(a);
    o[13] = __hiloint2double(0, (int)__float_as_uint(narrow32(a)));
    o[14] = (double)near32(a, ok);
    o[15] = ok ? 1.0 : 0.0;
}
extern "C" int run(const double *x, const double *z, double *out, long long n) {
    double *d = nullptr, *e = nullptr, *o = nullptr;
    cudaError_t r = cudaMalloc(&d, n * 8);
    if (r == cudaSuccess) r = cudaMalloc(&e, n * 8);
    if (r == cudaSuccess) r = cudaMalloc(&o, n * 128);
    if (r == cudaSuccess) r = cudaMemcpy(d, x, n * 8, cudaMemcpyHostToDevice);
    if (r == cudaSuccess) r = cudaMemcpy(e, z, n * 8, cudaMemcpyHostToDevice);
    if (r == cudaSuccess) k<<<(unsigned)((n + 255) / 256), 256>>>(d, e, o, n);
    if (r == cudaSuccess) r = cudaMemcpy(out, o, n * 128, cudaMemcpyDeviceToHost);
    cudaFree(d); cudaFree(e); cudaFree(o);
    return (int)r;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1711_11361_gb300 import build
    d = tmp_path_factory.mktemp("fp64")
    (d / "f.cu").write_text(SOURCE)
    # (the flags of the unit that uses the functions most)
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.COMMON, *build.UNITS["mb_sweep.cu"], "-I", build.CSRC,
                           "-shared", "-o", str(d / "f.so"), str(d / "f.cu")])
    lib = ctypes.CDLL(str(d / "f.so"))
    D = ctypes.POINTER(ctypes.c_double)
    lib.run.argtypes = [D, D, D, ctypes.c_longlong]

    def call(x, z=None):
        x = np.ascontiguousarray(x, dtype=np.float64)
        z = np.ascontiguousarray(x[::-1] if z is None else z, dtype=np.float64)
        out = np.empty((x.size, 16))
        assert lib.run(*(a.ctypes.data_as(D) for a in (x, z, out)), x.size) == 0
        return out
    return call


def _numbers(lo, hi, n, seed):
    """+-significand 2^e over every exponent lo .. hi - 1, and 2^hi; significands random, and next to 1, 2 and ties"""
    rng = np.random.default_rng(seed)
    m = 1.0 + rng.random(n)
    few = np.array([0.0, 1.0, 2.0, 3.0, 2.0 ** 28, 2.0 ** 29, 2.0 ** 29 + 1.0, 2.0 ** 30, 2.0 ** 52 - 1.0]) * 2.0 ** -52
    m[:n // 16] = 1.0 + rng.choice(few, n // 16)
    x = np.ldexp(m, rng.integers(lo, hi, n))
    x[::2] *= -1.0
    return np.concatenate([x, [2.0 ** lo, 2.0 ** hi, -2.0 ** hi]])


def _ulps(a, b):
    return np.max(np.abs(a.view(np.int64) - b.view(np.int64)))


def test_reciprocal(run):
    for seed in range(2):
        x = _numbers(-1021, 1021, 1 << 20, seed)
        o = run(x)
        assert np.max(np.abs(o[:, 1])) <= 1.01 * 2.0 ** -53
        assert _ulps(o[:, 0].copy(), o[:, 2].copy()) <= 1
    o = run(np.array([0.0, -0.0, np.nan, np.inf, -np.inf]))
    assert o[0, 0] == np.inf and o[1, 0] == -np.inf and np.isnan(o[2, 0])
    assert not np.any(np.isfinite(o[3:, 0]))     # (the comment promises no more of an infinity)


def test_square_root(run):
    for seed in range(2):
        x = np.abs(_numbers(-900, 1021, 1 << 20, seed))       # (the residual would lose its bits below)
        o = run(x)
        assert np.max(np.abs(o[:, 4]) / x) <= 2.0 * 1.51 * 2.0 ** -53
    x = np.abs(_numbers(-1021, 1021, 1 << 20, 7))
    o = run(x)
    assert _ulps(o[:, 3].copy(), o[:, 5].copy()) <= 2
    o = run(np.array([0.0, -1.0, -1e-300, np.nan]))
    assert o[0, 3] == 0.0 and np.all(np.isnan(o[1:, 3]))


SPECIAL = np.array([0.0, -0.0, np.inf, -np.inf, 5e-324, -5e-324, 2.0 ** -1022, -2.0 ** -1022, 1.0, -1.0, 1.7e308, -1.7e308])


def test_signs_and_order(run):
    x = np.concatenate([SPECIAL, [np.nan], _numbers(-1022, 1023, 4096, 3)])
    o = run(x)
    with np.errstate(invalid="ignore"):
        assert np.array_equal(o[:, 6], (x > 0).astype(float)) and np.array_equal(o[:, 7], (x >= 0).astype(float))
    a, b = (v.ravel() for v in np.meshgrid(x[~np.isnan(x)][:400], x[~np.isnan(x)][:400]))
    o = run(a, b)
    assert np.array_equal(o[:, 8], np.minimum(a, b)) and np.array_equal(o[:, 9], np.maximum(a, b))
    assert np.array_equal(o[:, 10], np.abs(a))


def test_twice_and_half(run):
    x = np.concatenate([[0.0, -0.0, np.inf, -np.inf, np.nan], _numbers(-1020, 1022, 1 << 16, 4)])
    o = run(x)
    assert np.array_equal(o[:, 11], 2.0 * x, equal_nan=True) and np.array_equal(o[:, 12], 0.5 * x, equal_nan=True)


def test_to_float(run):
    x = np.concatenate([SPECIAL, _numbers(-160, 140, 1 << 20, 5), np.ldexp(2.0 - 2.0 ** -25, np.arange(-130, 129)),
                        np.ldexp(1.0 + 2.0 ** -24, np.arange(-150, 128)), np.ldexp(1.0 + 3.0 * 2.0 ** -24, np.arange(-150, 128))])
    o = run(x)
    with np.errstate(over="ignore"):
        want = x.astype(np.float32)
    got = o[:, 13].copy().view(np.int64).astype(np.uint32)
    # (the unit flushes FP32 subnormals, which no state of use holds: as zero or as they are)
    normal = np.abs(want) >= np.float32(2.0 ** -126)
    assert np.array_equal(got[normal], want.view(np.uint32)[normal])
    assert np.all(np.abs(got[~normal].view(np.float32)) < np.float32(2.0 ** -126))
    # near32: to 2^-22 below 2^127, smaller than the least normal float as 0; the flag beyond
    small = np.abs(x) < 2.0 ** 127
    assert np.array_equal(o[:, 15] == 1.0, small)
    err = np.abs(o[small, 14] - x[small])
    assert np.all(err <= np.where(np.abs(x[small]) < 2.0 ** -126, np.abs(x[small]), 2.0 ** -22 * np.abs(x[small])))
