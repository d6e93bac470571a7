"""Quotient and root of the FP64 interaction terms (div_, root_ of engine.cuh) against CUDA's correctly rounded
operators: equal bit for bit, over the operands the terms can meet and the ones where a last-bit error would show."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1608_03722_gb300 import _build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "engine.cuh"
using namespace dsdna;
__global__ void k(const double* a, const double* b, long long n, double* out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += gridDim.x * (long long)blockDim.x) {
    out[i] = div_(a[i], b[i]);
    out[n + i] = __ddiv_rn(a[i], b[i]);
    out[2 * n + i] = root_(b[i]);
    out[3 * n + i] = __dsqrt_rn(b[i]);
  }
}
extern "C" int compare(const double* a, const double* b, long long n, double* out) {
  k<<<608, 256>>>(a, b, n, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("terms")
    (d / "terms.cu").write_text(SRC)
    so = str(d / "terms.so")
    subprocess.check_call([_build.nvcc(), *_build.ARCH, "-O3", "-std=c++17", "-I", _build.CSRC, "-shared", "-Xcompiler",
                           "-fPIC", str(d / "terms.cu"), "-o", so])
    return C.CDLL(so)


def _compare(lib, a, b):
    """Bits of (quotient, CUDA's, root, CUDA's)."""
    import torch
    ad, bd = (torch.tensor(x, dtype=torch.float64, device="cuda") for x in (a, b))
    out = torch.empty((4, len(a)), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.compare(C.c_void_p(ad.data_ptr()), C.c_void_p(bd.data_ptr()), C.c_longlong(len(a)),
                       C.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy()


def _ulps(x, k):
    return (x.view(np.int64) + k).view(np.float64)


def _operands(kind, rng, n):
    if kind == "separations":                      # squared lengths and products of the terms, 1e-12 .. 1e12
        return rng.choice([-1.0, 1.0], n) * 10.0 ** rng.uniform(-12, 12, n), 10.0 ** rng.uniform(-12, 12, n)
    if kind == "exponents":                        # quotients and operands up to 2^+-400
        return (rng.uniform(1, 2, n) * 2.0 ** rng.integers(-200, 200, n), rng.uniform(1, 2, n) * 2.0 ** rng.integers(-200, 200, n))
    if kind == "powers of two":                    # within 64 last bits of a power of two
        p = 2.0 ** rng.integers(-40, 40, (2, n))
        return _ulps(p[0], rng.integers(-64, 65, n)), _ulps(p[1], rng.integers(-64, 65, n))
    if kind == "one minus cosine squared":         # 1 - cs^2 down to its last bit
        return rng.uniform(-20, 20, n), rng.integers(1, 1 << 20, n) * 2.0 ** -53
    if kind == "extension limit":                  # r2 a few last bits below R0^2, and 1 - r2/R0^2
        c = rng.uniform(0.5, 9.0, n)
        return _ulps(c, -rng.integers(1, 1 << 12, n)), c
    if kind == "halfway":                          # quotients and roots next to the middle of two numbers
        b, q = rng.uniform(1, 2, n), rng.uniform(1, 4, n)
        t = q.astype(np.longdouble) * (1 + np.ldexp(np.longdouble(1), -53))
        half = n // 2
        b[half:] = _ulps((t * t).astype(np.float64), rng.integers(-2, 3, n))[half:]
        return _ulps((b.astype(np.longdouble) * t).astype(np.float64), rng.integers(-2, 3, n)), b
    raise KeyError(kind)


@pytest.mark.parametrize("kind", ["separations", "exponents", "powers of two", "one minus cosine squared",
                                  "extension limit", "halfway"])
def test_rounded_like_the_operators(lib, kind):
    rng = np.random.default_rng(17)
    for _ in range(4):
        a, b = _operands(kind, rng, 1 << 22)
        o = _compare(lib, a, b).view(np.int64)
        assert (o[0] == o[1]).all(), (kind, int((o[0] != o[1]).sum()))
        assert (o[2] == o[3]).all(), (kind, int((o[2] != o[3]).sum()))


def test_special_operands(lib):
    """Zeros, infinities, NaN, negative roots, and quotients beyond the largest number, as the operators give them."""
    v = np.array([0.0, -0.0, 1.0, -1.0, 2.5, -2.5, np.inf, -np.inf, np.nan, 1e300, -1e300, 1e-300, 2.0 ** 1000])
    a, b = (x.ravel() for x in np.meshgrid(v, v))
    keep = ~((np.abs(a) < 1e-100) & (np.abs(b) > 1e100) & np.isfinite(b) & (a != 0))   # quotients below the smallest normal number
    o = _compare(lib, a[keep], b[keep])
    for got, want in ((o[0], o[1]), (o[2], o[3])):
        assert ((got.view(np.int64) == want.view(np.int64)) | (np.isnan(got) & np.isnan(want))).all(), \
            [(x, y, g, w) for x, y, g, w in zip(a[keep], b[keep], got, want) if not (g == w or (np.isnan(g) and np.isnan(w)))]
