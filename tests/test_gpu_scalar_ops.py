"""The division and the widening of csrc/vanse_common.cuh over every kind of operand, compiled
into a small library of their own.

Reciprocal: the last Newton step rounds once the value r (2 - a r) of an r whose relative
error e is below 2^-20 (FP64, after the first step; e^2 then far below a rounding) or 2^-22
(FP32), so it is within half a unit plus 2^-21 of one of 1 / a, one unit at most from the
correctly rounded value; a product with it adds half a unit. Operands that the instruction
flushes or turns into zeros and infinities take the division, and agree with it exactly."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2409_02964_gb300", "csrc")
SOURCE = r"""
#include "vanse_common.cuh"
using namespace lbmv;
template <typename T>
__global__ void divide(const T* x, const T* a, T* rcp, T* quot, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    rcp[k] = rcp_nr(a[k]);
    quot[k] = Divisor<T>(a[k])(x[k]);
}
__global__ void widen_all(const float* a, double* out, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = widen(a[k]);
}
extern "C" int divide64(const double* x, const double* a, double* r, double* q, int n) {
    divide<double><<<(n + 255) / 256, 256>>>(x, a, r, q, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int divide32(const float* x, const float* a, float* r, float* q, int n) {
    divide<float><<<(n + 255) / 256, 256>>>(x, a, r, q, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int widen32(const float* a, double* out, int n) {
    widen_all<<<(n + 255) / 256, 256>>>(a, out, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2409_02964_gb300 import build
    d = tmp_path_factory.mktemp("ops")
    (d / "ops.cu").write_text(SOURCE)
    out = str(d / "libops.so")
    subprocess.run([build.nvcc(), build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + CSRC, "-o",
                    out, str(d / "ops.cu")], check=True)
    return ctypes.CDLL(out)


def _operands(dtype):
    """Random bit patterns (every exponent, subnormals, infinities, NaN), zeros, the edges of
    the normal range, and the values lattices divide by (phi, phi rho)."""
    bits = {np.float64: np.uint64, np.float32: np.uint32}[dtype]
    rng = np.random.default_rng(5)
    a = rng.integers(0, np.iinfo(bits).max, size=200000, dtype=bits, endpoint=True).view(dtype)
    fi = np.finfo(dtype)
    tiny, sub, big = fi.tiny, fi.smallest_subnormal, fi.max
    edge = [0.0, sub, 3 * sub, tiny / 4 + 7 * sub, tiny / 4, tiny / 2, tiny - sub, tiny, tiny + sub, 0.25 / tiny, 0.5 / tiny,
            1 / tiny, 2 / tiny, big, np.inf, np.nan, 1.0, 1 - fi.epsneg, 1 + fi.eps]
    edge = np.array(edge + [-v for v in edge], dtype=dtype)
    return np.concatenate([a, edge, rng.uniform(1e-6, 1.2, size=100000).astype(dtype)])


def _ulps(got, ref):
    """Distance in units of the last place (same-signed finite values); 0 where both are equal or NaN."""
    bits = {np.dtype(np.float64): np.int64, np.dtype(np.float32): np.int32}[got.dtype]
    same = (got == ref) | (np.isnan(got) & np.isnan(ref))
    d = np.abs(got.view(bits).astype(np.int64) - ref.view(bits).astype(np.int64))     # (wraps only where signs differ)
    ok = np.isfinite(got) & np.isfinite(ref) & (np.signbit(got) == np.signbit(ref))
    return np.where(same, 0.0, np.where(ok, d, np.inf))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_division(lib, dtype):
    import torch
    a = _operands(dtype)
    x = np.random.default_rng(6).permutation(a)
    x[: a.size // 2] = np.random.default_rng(7).normal(size=a.size // 2).astype(dtype)
    d = [torch.from_numpy(v).cuda() for v in (x, a, np.empty_like(a), np.empty_like(a))]
    fn = lib.divide64 if dtype == np.float64 else lib.divide32
    assert fn(*[ctypes.c_void_p(t.data_ptr()) for t in d], a.size) == 0
    rcp, quot = d[2].cpu().numpy(), d[3].cpu().numpy()
    with np.errstate(all="ignore"):
        want_r, want_q = dtype(1) / a, x / a
    mag, fi = np.abs(a), np.finfo(dtype)
    normal = (mag >= fi.tiny) & (mag < 1 / fi.tiny)      # a and 1 / a normal
    off = _ulps(rcp, want_r)
    assert off[normal].max() <= 1
    assert off[~normal].max() == 0
    off = _ulps(quot, want_q)
    assert off[~normal].max() == 0
    plain = normal & (np.abs(want_q) >= 2 * fi.tiny) & np.isfinite(want_q) & (np.abs(want_q) <= fi.max / 2)
    assert off[plain].max() <= 2


def test_widening(lib):
    import torch
    a = _operands(np.float32)
    t, o = torch.from_numpy(a).cuda(), torch.empty(a.size, dtype=torch.float64, device="cuda")
    assert lib.widen32(ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(o.data_ptr()), a.size) == 0
    with np.errstate(invalid="ignore"):
        got, want = o.cpu().numpy(), a.astype(np.float64)
    nan = np.isnan(want)
    assert np.isnan(got[nan]).all()
    assert np.array_equal(got[~nan].view(np.int64), want[~nan].view(np.int64))
