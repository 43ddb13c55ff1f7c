"""The FP64 step kernels' quotients (GPU): recip (csrc/flb_internal.cuh) and d1q3_quotient
(csrc/d1q3_common.cuh) against exact division, over the exponent range and at the edges where they
branch to CUDA's division: magnitudes outside 2^-100 .. 2^100, zeros, infinities, NaN, and for the D1Q3
quotient negative populations (the FP32 estimate of their sum could cancel).

Tolerance where the FP32 estimate is used, relative to the quotient:
  recip: |e| = |1 - a y| <= 2^-22 (narrowing 2^-23, hardware reciprocal 2^-23), the series ends with e^3 <= 2^-66,
      one rounding: 2^-53 + 2^-65
  d1q3_quotient: |e| <= 2^-21.4 (three narrowed values, two FP32 additions, reciprocal), e^3 <= 2^-64, two
      roundings: 2^-52 + 2^-63
Elsewhere equal bit for bit to IEEE division."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_1010_1233_gb300 import build as B

pytestmark = pytest.mark.gpu
LD = np.longdouble

SOURCE = r"""
#include "d1q3_common.cuh"
__global__ void k(const double* a, int n, double* r) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) r[i] = flb::recip(a[i]);
}
__global__ void q(const double* g, const double* num, int n, double* r) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double g0 = g[i], g1 = g[n + i], g2 = g[2 * n + i];
    r[i] = flb::d1q3_quotient(num[i], __dadd_rn(g0, __dadd_rn(g1, g2)), g0, g1, g2);
  }
}
extern "C" int run_recip(const double* a, int n, double* r) { k<<<64, 256>>>(a, n, r); return cudaDeviceSynchronize(); }
extern "C" int run_quot(const double* g, const double* num, int n, double* r) { q<<<64, 256>>>(g, num, n, r); return cudaDeviceSynchronize(); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotients")
    (d / "q.cu").write_text(SOURCE)
    subprocess.run([B.nvcc_path(), B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC",
                    "-I", B.INCLUDE, "-I", B.CSRC, str(d / "q.cu"), "-o", str(d / "q.so")], check=True)
    return ctypes.CDLL(str(d / "q.so"))


def _call(f, *arrays):
    n = arrays[-1].size
    t = [torch.tensor(a, dtype=torch.float64, device="cuda").contiguous() for a in arrays]
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(x.data_ptr()) for x in t]
    assert f(*p, n, ctypes.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy()


def _ordinary(x):
    return (np.abs(x) >= 2.0 ** -100) & (np.abs(x) < 2.0 ** 100)


EDGES = [s * v for s in (1, -1) for k in (-1074, -1022, -101, -100, -99, -1, 0, 1, 99, 100, 101, 1023)
         for v in (2.0 ** k, np.nextafter(2.0 ** k, 0), np.nextafter(2.0 ** k, np.inf))]
EDGES += [0.0, -0.0, np.inf, -np.inf, np.nan, np.finfo(float).max]


def test_reciprocal(lib):
    rng = np.random.default_rng(1)
    a = np.concatenate([EDGES, rng.uniform(0.5, 2, 100_000), rng.choice([-1, 1], 100_000) * np.exp2(rng.uniform(-110, 110, 100_000)),
                        1 + np.arange(-2000, 2000) * 2.0 ** -52, 1 + np.arange(-2000, 2000) * 2.0 ** -23])
    r = _call(lib.run_recip, a)
    with np.errstate(all="ignore"):
        exact = 1.0 / a
    fast = _ordinary(a)
    assert np.array_equal(r[~fast], exact[~fast], equal_nan=True)
    err = np.abs(r[fast].astype(LD) * a[fast].astype(LD) - 1)
    assert err.max() <= LD(2) ** -53 + LD(2) ** -65, float(err.max() * 2.0 ** 53)


def test_d1q3_quotient(lib):
    rng = np.random.default_rng(2)
    n = 100_000
    near = np.stack([2 / 3 + 0.2 * rng.standard_normal(n), 1 / 6 + 0.1 * rng.standard_normal(n),
                     1 / 6 + 0.1 * rng.standard_normal(n)])                     # some negative, some sums near zero
    wide = rng.choice([-1, 1, 1, 1], (3, n)) * np.exp2(rng.uniform(-110, 110, (3, n)))
    e = np.array(EDGES)
    c = lambda v: np.full_like(e, v)
    one = np.stack([np.stack([e, c(1 / 6), c(1 / 6)]), np.stack([c(2 / 3), e, c(0.25)]), np.stack([c(2 / 3), c(0.25), e]),
                    np.stack([e, -e, c(1)]), np.stack([e, e, e])], 1).reshape(3, -1)
    g = np.concatenate([near, wide, one], 1)
    with np.errstate(all="ignore"):
        j, rho = g[1] - g[2], g[0] + (g[1] + g[2])
        g, num = np.concatenate([g, g], 1), np.concatenate([j * j, j])
        rho = np.concatenate([rho, rho])
        exact = num / rho
    r = _call(lib.run_quot, g, num)
    fast = (_ordinary(g) & (g > 0)).all(0)
    assert 0.3 < fast.mean() < 0.9
    assert np.array_equal(r[~fast], exact[~fast], equal_nan=True)
    zero = fast & (num == 0)
    assert (r[zero] == 0).all()
    fast &= num != 0
    assert np.isfinite(r[fast]).all()
    err = np.abs(r[fast].astype(LD) * rho[fast].astype(LD) / num[fast].astype(LD) - 1)
    assert err.max() <= LD(2) ** -52 + LD(2) ** -63, float(err.max() * 2.0 ** 53)
