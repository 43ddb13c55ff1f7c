"""Fixed-point FP64 normals (csrc/normals64.cuh) against extended precision.

The header also compiles as plain C++, so the edges of its reductions (words at powers of
two, table boundaries, the largest and smallest uniforms) are checked on the CPU; the GPU
test draws through flb_philox, where the square root starts from the hardware estimate.

Tolerance: half an ulp of the result for the final rounding, 2^-56 for the fixed-point
terms (each carries a few units of 2^-59 in the angle and, for ua < 1/2, in -ln ua, whose
root r >= 1.17 does not amplify it), and 2^-60 / r for ua >= 1/2, where -ln ua has units of
2^-63 and r may be small.
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
    wa, wb = wa.astype(LD), wb.astype(LD)
    r = np.sqrt(-2 * np.log((wa + LD(0.5)) * LD(2) ** -32))
    # the angle reduced exactly to (-1/8, 1/8] turns around a multiple of a quarter turn
    x = 2 * wb + 1                                    # units of 2^-33 turns
    k = np.floor(x / LD(2) ** 31 + LD(0.5))
    a = TWO_PI * ((x - k * LD(2) ** 31) * LD(2) ** -33)
    c, s, k = np.cos(a), np.sin(a), k.astype(int) % 4
    c, s = np.choose(k, [c, -s, -c, s]), np.choose(k, [s, c, -s, -c])
    for n, want in ((n0, r * c), (n1, r * s)):
        tol = 0.5 * np.spacing(np.abs(n)) + 2.0 ** -56 + (2.0 ** -60 / r).astype(float)
        err = np.abs(n.astype(LD) - want)
        i = int(np.argmax(err / tol))
        assert (err <= tol).all(), (int(wa[i]), int(wb[i]), float(err[i]), float(tol[i]))


def test_edges_on_the_cpu(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "n.cpp"
    src.write_text('#include "normals64.cuh"\nextern "C" void f(const uint32_t* a, const uint32_t* b, double* o, int n) {'
                   "for (int i = 0; i < n; ++i) flb::fx_box_muller(a[i], b[i], o[2 * i], o[2 * i + 1]); }\n")
    so = tmp_path / "n.so"
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", B.CSRC, str(src), "-o", str(so)], check=True)
    edge = [(1 << i) + d for i in range(32) for d in (-2, -1, 0, 1)] + [2**32 - (1 << i) + d for i in range(32)
                                                                         for d in (-1, 0, 1)]
    edge += [(i << 25) // 2 + d for i in range(256) for d in (-1, 0, 1)]
    edge = np.unique(np.array(edge, dtype=np.int64) & 0xFFFFFFFF).astype(np.uint32)
    rnd = np.random.default_rng(3).integers(0, 2**32, (2, 100_000), dtype=np.uint64).astype(np.uint32)
    wa = np.concatenate([np.repeat(edge, len(edge)), rnd[0]])
    wb = np.concatenate([np.tile(edge, len(edge)), rnd[1]])
    out = np.empty((len(wa), 2))
    p = lambda x, t: x.ctypes.data_as(ctypes.POINTER(t))
    ctypes.CDLL(str(so)).f(p(wa, ctypes.c_uint32), p(wb, ctypes.c_uint32), p(out, ctypes.c_double), len(wa))
    _check(wa, wb, out[:, 0], out[:, 1])


@pytest.mark.gpu
def test_drawn_normals_on_the_gpu():
    from paper_1010_1233_gb300 import philox
    words, n = philox(np.arange(400_000, dtype=np.uint32), 3, 1, 0, 2, 77)
    _check(words[:, 0], words[:, 1], n[:, 0], n[:, 1])
    _check(words[:, 2], words[:, 3], n[:, 2], n[:, 3])
