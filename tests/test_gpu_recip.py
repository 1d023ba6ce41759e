"""The dense solver's reciprocal, reciprocal root and root (csrc/recip64.cuh) against quadruple
precision and against CUDA's own operations: random mantissas at every exponent, powers of two, values
next to 1, the ends of the range that the approximate instructions serve, subnormal numbers, zero,
infinity and NaN.

Bounds, in units of the last place of the result (derived in the header): 9/16 for the reciprocal, 5/4
for the reciprocal root, 1/2 (and a thousandth for the second-order rest) for the root.  Outside the range
the ordinary operations' results, bit for bit.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2507_08578_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "recip64.cuh"
__global__ void k(const double* x, double* y, long long n) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i], a = fabs(v), r = kss::fast_rsqrt(a);
  y[i] = kss::fast_rcp(v);
  y[n + i] = r;
  y[2 * n + i] = kss::sqrt_from(a, r);
  y[3 * n + i] = 1.0 / v;
  y[4 * n + i] = 1.0 / sqrt(a);
  y[5 * n + i] = sqrt(a);
  y[6 * n + i] = kss::mid_range(v);
}
extern "C" int run(const double* x, double* y, long long n) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


def values():
    rng = np.random.default_rng(12)
    ex = np.repeat(np.arange(-1074, 1024), 60)
    x = [np.ldexp(1.0 + rng.random(ex.size), ex - 1) * np.where(rng.random(ex.size) < 0.5, -1.0, 1.0)]
    x.append(1.0 + rng.random(60000))
    x.append(4.0 * rng.random(60000))
    x.append(np.ldexp(1.0, np.arange(-1074, 1024)))
    one = np.ones(1).view(np.int64)[0]
    x.append((one + np.arange(-2000, 2000)).view(np.float64))
    for e in (-927, 913):  # the ends of the range
        end = np.full(1, np.ldexp(1.0, e)).view(np.int64)[0]
        x.append((end + np.arange(-50, 50)).view(np.float64))
    x.append(np.arange(1, 50, dtype=np.int64).view(np.float64))  # the smallest subnormal numbers
    x.append(np.array([0.0, -0.0, np.inf, -np.inf, np.nan, np.finfo(float).max, np.finfo(float).tiny]))
    return np.concatenate(x)


def test_against_quadruple_precision_and_cuda(tmp_path):
    import torch
    src, so = tmp_path / "r.cu", tmp_path / "r.so"
    src.write_text(SRC)
    subprocess.run([B.nvcc(), *B.ARCH, *B.COMMON, "-shared", str(src), "-o", str(so)], check=True)
    x = values()
    tx = torch.from_numpy(x).cuda()
    ty = torch.empty(7, x.size, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    run = ctypes.CDLL(str(so)).run
    run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]
    assert run(tx.data_ptr(), ty.data_ptr(), x.size) == 0
    rcp, rsq, root, c_rcp, c_rsq, c_root, mid = ty.cpu().numpy()
    a = np.abs(x)
    inside = (a >= 2.0 ** -927) & (a < 2.0 ** 913)
    assert np.array_equal(mid != 0, inside)
    for got, own in ((rcp, c_rcp), (rsq, c_rsq), (root, c_root)):
        assert np.array_equal(got[~inside].view(np.int64), own[~inside].view(np.int64))
    # at least 11 bits beyond double
    assert np.finfo(np.longdouble).nmant >= 63
    q = x[inside].astype(np.longdouble)
    s = np.sqrt(np.abs(q))
    for got, own, exact, bound in ((rcp, c_rcp, 1 / q, 0.5625), (rsq, c_rsq, 1 / s, 1.25), (root, c_root, s, 0.501)):
        ulp = np.spacing(np.abs(exact).astype(np.float64))
        err = np.max(np.abs(got[inside] - exact) / ulp)
        assert err <= bound, err
        assert np.max(np.abs(got[inside] - own[inside]) / ulp) <= 2
