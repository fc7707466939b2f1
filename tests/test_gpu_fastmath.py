"""The short FP64 reciprocal, reciprocal square root and float -> double
conversion (fastmath.cuh) over their whole range, against exact residuals and
CUDA's own functions."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "fastmath.cuh"
// out: rcp(x), 1 - x rcp(x), 1 / x, rsq(x), 1 - x rsq(x)^2, rsqrt(x); residuals
// from exact products (the error of a product by fma), rounded once at the end
__global__ void k(const double *x, long n, double *out) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const double a = x[i], r = hff::rcp(a), s = hff::rsq(a), p = s * s, pe = fma(s, s, -p);
    double *o = out + 6 * i;
    o[0] = r; o[1] = fma(-a, r, 1.0); o[2] = 1.0 / a;
    o[3] = s; o[4] = fma(-a, p, 1.0) - a * pe; o[5] = rsqrt(a);
  }
}
__global__ void kc(unsigned first, long n, unsigned long long *bad) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    const float f = __uint_as_float(first + (unsigned)i);
    const double a = hff::to_double(f), b = (double)f;
    if (!(__double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b))) atomicAdd(bad, 1ull);
  }
}
extern "C" int run(const double *x, long n, double *out) { k<<<1024, 256>>>(x, n, out); return (int)cudaDeviceSynchronize(); }
extern "C" int conv(unsigned first, long n, unsigned long long *bad) { kc<<<4096, 256>>>(first, n, bad); return (int)cudaDeviceSynchronize(); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2406_14512_gb300 import build
    d = tmp_path_factory.mktemp("fastmath")
    (d / "t.cu").write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.SRC, "-shared", "-o", str(d / "t.so"), str(d / "t.cu")],
                   check=True, capture_output=True)
    return C.CDLL(str(d / "t.so"))


def _run(lib, x):
    import torch
    xd = torch.from_numpy(np.ascontiguousarray(x, np.float64)).cuda()
    out = torch.empty(len(x), 6, dtype=torch.float64, device="cuda")
    assert lib.run(C.c_void_p(xd.data_ptr()), C.c_long(len(x)), C.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy().T


def test_reciprocal_and_root_in_the_middle_of_the_range(lib):
    """Exponents that take the short forms (2^-985 to 2^985 kept clear of both
    ends).  rcp: the series ends below 2^-75, one rounding is left: 2^-53 of the
    value, like 1 / x, and a thousandth more for the rounding of the residual
    itself.  rsq: one rounding and the remainder, below (5/16) 2^-54 for an e of
    2^-18, the residual 1 - x y^2 twice their sum: 1.16 times 2^-52 (CUDA's rsqrt
    may be off by an ulp, 2 times 2^-52).  Mantissas at random, all 2^16 leading ones,
    and neighbours of powers of two, where an ulp changes its size."""
    rng = np.random.default_rng(1)
    m = np.concatenate([rng.random(4_000_000) + 1.0, 1.0 + np.arange(65536) / 65536.0, 1.0 + np.arange(64) * 2.0 ** -52,
                        2.0 - np.arange(1, 65) * 2.0 ** -52])
    e = rng.integers(-985, 985, len(m))
    e[4_000_000:] = np.tile([0, 1], len(m))[:len(m) - 4_000_000]
    r, rr, inv, s, sr, root = _run(lib, np.ldexp(m, e))
    assert np.abs(rr).max() <= 1.001 * 2.0 ** -53, np.abs(rr).max() * 2.0 ** 53
    assert np.abs(sr).max() <= 1.16 * 2.0 ** -52, np.abs(sr).max() * 2.0 ** 52
    assert (np.abs(r - inv) <= np.spacing(inv)).all() and (np.abs(s - root) <= 2 * np.spacing(root)).all()
    r, rr, inv, *_ = _run(lib, -np.ldexp(m, e))
    assert np.abs(rr).max() <= 1.001 * 2.0 ** -53 and (np.abs(r - inv) <= np.spacing(np.abs(inv))).all()


def test_ends_of_the_range(lib):
    """Both sides of the limits of the short forms, subnormals, zero, infinity and
    NaN: as CUDA's functions, to the last bit outside the short forms."""
    e = np.concatenate([np.arange(-1074, -985), np.arange(985, 1024)])
    x = np.concatenate([np.ldexp(1.0, e), np.ldexp(1.75, e[e > -1070]), np.ldexp(1.0, e[e > -1070]) * (1 - 2.0 ** -53),
                        [0.0, np.inf, np.nan, 5e-324]])
    with np.errstate(all="ignore"):
        r, _, inv, s, _, root = _run(lib, x)
        field = (x.view(np.uint64) >> np.uint64(52)) & np.uint64(0x7ff)
        out = (field < 32) | (field >= 2047 - 32)
        assert out.sum() > 150 and (~out).sum() > 30
        for got, want in ((r, inv), (s, root)):
            same = (got == want) | (np.isnan(got) & np.isnan(want))
            assert same[out].all()
            assert (same | (np.abs(got - want) <= 2 * np.spacing(np.abs(want)))).all()
        r, _, inv, *_ = _run(lib, np.concatenate([-x[:-4], [-0.0, -np.inf]]))
        assert ((r == inv) | (np.abs(r - inv) <= np.spacing(np.abs(inv)))).all()


def test_every_float_converts_as_the_hardware_does(lib):
    import torch
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    assert lib.conv(C.c_uint(0), C.c_long(1 << 32), C.c_void_p(bad.data_ptr())) == 0
    assert int(bad.item()) == 0
