"""The kernels' own reciprocals and quotients against CUDA's, over every exponent: random fractions, the
fractions next to powers of two, zeros, subnormals, infinities, NaN."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "xk_recip.cuh"
__global__ void k64(const double *x, long long n, double *a, double *b, double *c, double *r)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        a[i] = xk::reciprocal64(x[i]);
        b[i] = xk::reciprocal_rn(x[i]);
        c[i] = xk::reciprocal_newton(x[i]);
        r[i] = 1.0 / x[i];
    }
}
__global__ void kover(const double *x, const double *d, long long n, double *a, double *r)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        a[i] = xk::over(x[i], d[i], xk::reciprocal_rn(d[i]));
        r[i] = x[i] / d[i];
    }
}
__global__ void k32(const float *x, long long n, float *a, float *r)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        a[i] = xk::reciprocal32(x[i]);
        r[i] = 1.0f / x[i];
    }
}
extern "C" int run64(const double *x, long long n, double *a, double *b, double *c, double *r)
{
    k64<<<1024, 256>>>(x, n, a, b, c, r);
    return cudaDeviceSynchronize();
}
extern "C" int run_over(const double *x, const double *d, long long n, double *a, double *r)
{
    kover<<<1024, 256>>>(x, d, n, a, r);
    return cudaDeviceSynchronize();
}
extern "C" int run32(const float *x, long long n, float *a, float *r)
{
    k32<<<1024, 256>>>(x, n, a, r);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2512_06729_gb300 import build as xkbuild
    d = tmp_path_factory.mktemp("recip")
    src, out = d / "recip.cu", d / "librecip.so"
    src.write_text(SOURCE)
    subprocess.run([xkbuild.nvcc(), *xkbuild.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-I", xkbuild.CSRC, str(src), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


def _call(fn, *arrays):
    """fn over device copies of the given arrays, whose last ones are results."""
    dev = [torch.as_tensor(a).cuda() for a in arrays]
    n = ctypes.c_longlong(len(arrays[0]))
    args = [ctypes.c_void_p(t.data_ptr()) for t in dev]
    torch.cuda.synchronize()
    assert fn(args, n) == 0
    return [t.cpu().numpy() for t in dev]


def _every_exponent(ebits, fbits, uint, per, rng):
    """Bit patterns: for every exponent and both signs, `per` random fractions and the extreme ones."""
    expo = np.arange(1 << ebits, dtype=uint)
    frac = rng.integers(0, 1 << fbits, size=(1 << ebits, per), dtype=uint)
    ends = np.array([0, 1, 2, (1 << fbits) - 1, (1 << fbits) - 2, 1 << (fbits - 1), (1 << (fbits - 1)) - 1], dtype=uint)
    frac = np.concatenate([frac, np.tile(ends, (1 << ebits, 1))], axis=1)
    u = ((expo[:, None] << uint(fbits)) | frac).ravel()
    return np.concatenate([u, u | (uint(1) << uint(ebits + fbits))])


def _units(a, b, kind):
    """Units in the last place between a and b of the same sign; NaN agrees with NaN only."""
    nan = np.isnan(a) & np.isnan(b)
    ia, ib = a.view(kind), b.view(kind)
    same = (ia >= 0) == (ib >= 0)
    return np.where(nan, 0, np.where(same & ~np.isnan(a) & ~np.isnan(b), np.abs(ia - ib), 1 << 30))


def test_fp64_reciprocals(lib):
    x = _every_exponent(11, 52, np.uint64, 500, np.random.default_rng(1)).view(np.float64)
    z = np.zeros_like(x)
    _, series, rounded, newton, want = _call(lambda p, n: lib.run64(p[0], n, *p[1:]), x, z, z, z, z)
    assert np.max(_units(rounded, want, np.int64)) == 0
    assert np.max(_units(series, want, np.int64)) <= 1
    assert np.max(_units(newton, want, np.int64)) <= 1


def test_fp64_quotients(lib):
    rng = np.random.default_rng(2)
    every = _every_exponent(11, 52, np.uint64, 100, rng).view(np.float64)
    pairs = [(rng.permutation(every), rng.permutation(every))]
    # quotients near one, near the ends of the exponents for which the product is taken, of subnormals
    for ex, ed in ((1023, 1023), (515, 515), (1530, 1530), (515, 1530), (1530, 515), (514, 1023), (1531, 1023), (1023, 514),
                   (1023, 1531), (0, 0), (1, 1), (0, 1), (0, 1023), (2046, 1), (1, 2046)):
        n = 20000
        make = lambda e: ((np.uint64(e) << np.uint64(52)) | rng.integers(0, 1 << 52, n, dtype=np.uint64)).view(np.float64)
        pairs.append((make(ex), make(ed)))
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308, 1.0, 0.3])
    pairs.append(tuple(a.ravel() for a in np.meshgrid(special, special)))
    x, d = (np.concatenate([p[i] for p in pairs]) for i in range(2))
    z = np.zeros_like(x)
    _, _, got, want = _call(lambda p, n: lib.run_over(p[0], p[1], n, *p[2:]), x, d, z, z)
    assert np.max(_units(got, want, np.int64)) == 0


def test_fp32_reciprocal(lib):
    x = _every_exponent(8, 23, np.uint32, 20000, np.random.default_rng(3)).view(np.float32)
    z = np.zeros_like(x)
    _, got, want = _call(lambda p, n: lib.run32(p[0], n, *p[1:]), x, z, z)
    assert np.max(_units(got, want, np.int32)) <= 1
