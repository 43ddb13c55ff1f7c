"""Fixed-point FP64 normals (csrc/normals64.cuh) where the radius is small: ua near 1, r = sqrt(-2 ln ua)
down to 1.5e-5.

Tolerance: half an ulp of the result for the final rounding, and for the fixed-point terms
  ua >= 1 - 2^-8 (the logarithm keeps its leading zeros: a few units of 2^-61 of its own size, half that
      in r; sine and cosine a few of 2^-62 of r): 2^-57 r,
  otherwise 2^-56 (-ln ua in units of 2^-63 or 2^-59 over r >= 0.088 or 1.17; the angle's terms times r).
"""
import ctypes
import shutil
import subprocess

import numpy as np
import pytest

from paper_1010_1233_gb300 import build as B

LD = np.longdouble
TWO_PI = LD("6.283185307179586476925286766559005768394")


def _check(wa, wb, n0, n1):
    d = (2.0 ** 32 - 0.5 - wa.astype(LD)) * LD(2) ** -32            # 1 - ua, exact
    r = np.sqrt(-2 * np.log1p(-d))
    x = 2 * wb.astype(LD) + 1                                        # the angle in units of 2^-33 turns
    k = np.floor(x / LD(2) ** 31 + LD(0.5))
    a = TWO_PI * ((x - k * LD(2) ** 31) * LD(2) ** -33)
    c, s, k = np.cos(a), np.sin(a), k.astype(int) % 4
    c, s = np.choose(k, [c, -s, -c, s]), np.choose(k, [s, c, -s, -c])
    fixed = np.where(d < 2.0 ** -8, 2.0 ** -57 * r.astype(float), 2.0 ** -56)
    for n, want in ((n0, r * c), (n1, r * s)):
        tol = 0.5 * np.spacing(np.abs(n)) + fixed
        err = np.abs(n.astype(LD) - want).astype(float)
        i = int(np.argmax(err / tol))
        assert (err <= tol).all(), (int(wa[i]), int(wb[i]), float(err[i]), float(tol[i]))


def _words():
    """Words of ua near 1 over all scales of 1 - ua, and around the boundary of the last table entry."""
    rng = np.random.default_rng(11)
    one = [2 ** 32 - 1 - i for i in range(64)] + [2 ** 32 - (1 << i) + d for i in range(1, 32) for d in (-2, -1, 0, 1)]
    one += [2 ** 32 - 2 ** 24 + d for d in range(-40, 40)] + [2 ** 31 + d for d in range(-4, 5)]
    one += [2 ** 32 - 1 - int(2 ** e) for e in rng.uniform(0, 31, 4000)]
    wa = np.array(one, dtype=np.int64).astype(np.uint32)
    wb = rng.integers(0, 2 ** 32, len(wa), dtype=np.uint64).astype(np.uint32)
    edge = np.array([0, 1, 2 ** 29, 2 ** 30 - 1, 2 ** 30, 2 ** 31 - 1, 2 ** 31, 3 * 2 ** 30, 2 ** 32 - 1], dtype=np.uint32)
    return (np.concatenate([wa, np.repeat(wa[:300], len(edge))]), np.concatenate([wb, np.tile(edge, 300)]))


def test_small_radii_on_the_cpu(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "n.cpp"
    src.write_text('#include "normals64.cuh"\nextern "C" void f(const uint32_t* a, const uint32_t* b, double* o, int n) {'
                   "for (int i = 0; i < n; ++i) flb::fx_box_muller(a[i], b[i], o[2 * i], o[2 * i + 1]); }\n")
    so = tmp_path / "n.so"
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", B.CSRC, str(src), "-o", str(so)], check=True)
    wa, wb = _words()
    out = np.empty((len(wa), 2))
    p = lambda x, t: x.ctypes.data_as(ctypes.POINTER(t))
    ctypes.CDLL(str(so)).f(p(wa, ctypes.c_uint32), p(wb, ctypes.c_uint32), p(out, ctypes.c_double), len(wa))
    _check(wa, wb, out[:, 0], out[:, 1])


@pytest.mark.gpu
def test_small_radii_on_the_gpu():
    # the drawn pairs whose first word is near 2^32 (one in 256 has ua >= 1 - 2^-8)
    from paper_1010_1233_gb300 import philox
    words, n = philox(np.arange(3_000_000, dtype=np.uint32), 3, 1, 0, 2, 77)
    for q in (0, 2):
        near = words[:, q] >= 2 ** 32 - 2 ** 25
        assert near.sum() > 10_000
        _check(words[near, q], words[near, q + 1], n[near, q], n[near, q + 1])
