"""The FP64 reciprocal and square root of the tile kernels against IEEE division and
sqrt, over the whole range of exponents and at the exponents where they hand over.

The hardware's approximations are held to 2^-18 first (d below).  The reciprocal's two
Newton steps then leave d^4 = 2^-72 before the one rounding of the result, the root's
iteration 1.5 (1.5 d^2)^2 = 2^-70: a result differs from the correctly rounded one only
where the exact value lies that close to the middle of two doubles (2^-54 wide halves),
in at most 2^-17 and 2^-15 of random arguments, and then by one unit in the last place.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm.h"
#include "lbm_internal.h"
#include "lbm_kernels.cuh"
__global__ void math(const double* v, double* inv, double* root, double* rcp, double* rsq, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        inv[i] = lbm::inv64(v[i]);
        root[i] = lbm::root64(v[i]);
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(rcp[i]) : "d"(v[i]));
        asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(rsq[i]) : "d"(v[i]));
    }
}
extern "C" int run(const double* v, double* inv, double* root, double* rcp, double* rsq, long long n) {
    math<<<1024, 256>>>(v, inv, root, rcp, rsq, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    from paper_2402_15752_gb300 import build
    d = tmp_path_factory.mktemp("fp64_math")
    src, lib = str(d / "math.cu"), str(d / "libmath.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc()] + build.NVCC_FLAGS + ["-shared", src, "-o", lib], check=True)
    L = ctypes.CDLL(lib)

    def call(v):
        x = torch.from_numpy(np.ascontiguousarray(v)).cuda()
        out = [torch.empty_like(x) for _ in range(4)]
        torch.cuda.synchronize()
        p = [ctypes.c_void_p(t.data_ptr()) for t in [x] + out]
        assert L.run(*p, ctypes.c_longlong(x.numel())) == 0
        return [t.cpu().numpy() for t in out]
    return call


def _bits(exponents, mantissas, negative=0):
    e, m = np.asarray(exponents, np.uint64), np.asarray(mantissas, np.uint64)
    return ((np.uint64(negative) << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)


def _mantissas(rng, n):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    m[:8] = [0, 1, 2, (1 << 52) - 1, (1 << 52) - 2, 1 << 51, (1 << 51) - 1, (1 << 51) + 1]
    return m


def _off(got, want):
    """Distance in units in the last place (finite values of one sign)."""
    return np.abs(got.view(np.int64) - want.view(np.int64))


def test_the_hardware_approximations(run):
    # every leading 20 bits of the significand, at both parities of the exponent
    hi = np.arange(1 << 20, dtype=np.uint64) << np.uint64(32)
    low = np.random.default_rng(1).integers(0, 1 << 32, 1 << 20, dtype=np.uint64)
    v = np.concatenate([_bits(np.full(1 << 20, e), hi | l) for e in (1022, 1023) for l in (np.uint64(0), low)])
    _, _, rcp, rsq = run(v)
    assert np.abs(rcp * v - 1.0).max() < 2.0 ** -18
    assert np.abs(rsq * np.sqrt(v) - 1.0).max() < 2.0 ** -18


@pytest.mark.parametrize("negative", [0, 1])
def test_reciprocal(run, negative):
    rng = np.random.default_rng(2 + negative)
    n = 1 << 24
    e = rng.integers(1, 2046, n, dtype=np.uint64)  # 1 / b stays normal
    v = _bits(e, _mantissas(rng, n), negative)
    inv = run(v)[0]
    off = _off(inv, 1.0 / v)
    assert off.max() <= 1
    assert np.count_nonzero(off) <= n * 2.0 ** -17


def test_square_root(run):
    rng = np.random.default_rng(4)
    n = 1 << 24
    v = _bits(rng.integers(0x036, 2047, n, dtype=np.uint64), _mantissas(rng, n))
    root = run(v)[1]
    off = _off(root, np.sqrt(v))
    assert off.max() <= 1
    assert np.count_nonzero(off) <= n * 2.0 ** -15


def test_the_hand_over_exponents_and_special_values(run):
    rng = np.random.default_rng(5)
    m = _mantissas(rng, 4096)
    with np.errstate(all="ignore"):
        for e in (0x035, 0x036, 0x037, 0x7c7, 0x7c8, 0x7c9, 1, 2, 2045):
            v = _bits(np.full(m.size, e), m)
            inv, root = run(v)[:2]
            assert _off(inv, 1.0 / v).max() <= 1, hex(e)
            # the caller adds 1e-4
            assert _off(root + 1e-4, np.sqrt(v) + 1e-4).max() <= 1, hex(e)
        v = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -np.nan, 5e-324, -5e-324, 1e-310, -1.0])
        inv, root = run(v)[:2]
        np.testing.assert_array_equal(inv, 1.0 / v)
        want = np.where(v < 1e-300, np.where(v < 0, np.nan, 0.0), np.sqrt(v))
        np.testing.assert_array_equal(root, want)
