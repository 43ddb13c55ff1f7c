"""Sampling passes at the edges of their block split (GPU): groups of row pairs that do not fill
a block, one field of one row, column tiles past the last column, tiles cut down to single
sectors and field pairs dealt to several blocks, one-pass columns of the column-tiled spectrum,
against numpy's FFT in FP64.

Tolerance: a transform of V points has a relative error of ~log2(V) roundings in the root
mean square over its points; products double it: 4 log2(V) eps of the largest sum."""
import numpy as np
import pytest
import torch

from paper_1010_1233_gb300 import Sim, workloads as W
from paper_1010_1233_gb300.sim import spectra_accumulate, unpack_pair_sums

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("F,ny,nx", [(1, 1, 2), (1, 2, 4), (3, 1, 8), (1, 8, 16), (5, 2, 256), (9, 256, 256),
                                     (2, 64, 512), (11, 32, 64), (3, 1, 2048), (3, 1024, 64), (1, 4, 1024),
                                     (3, 64, 4096), (2, 256, 4096), (2, 16, 8192)])
def test_pair_sums_match_fft(precision, F, ny, nx):
    dt, eps = (torch.float64, 2.0 ** -53) if precision == "fp64" else (torch.float32, 2.0 ** -24)
    x = torch.tensor(W.random_perturbation((F, ny, nx), F + ny + nx), dtype=dt, device="cuda")
    sums, mean0 = spectra_accumulate(x)
    sums, mean0 = spectra_accumulate(x, sums, mean0)
    k = np.fft.rfft2(x.double().cpu().numpy())
    tol = 4 * max(np.log2(nx * ny), 1) * eps
    for (a, b), g in unpack_pair_sums(sums, F, ny, nx).items():
        want = 2 * k[a] * k[b].conj()
        scale = np.sqrt(np.abs(k[a]).max() * np.abs(k[b]).max()) ** 2 * 2
        assert np.abs(g - want).max() <= tol * scale, (a, b)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_uneven_batch_equals_single_runs(precision):
    # the split follows the whole batch; a replica's sums do not
    reps = [W.replica("D2Q9", nx, ny, W.taus_d2q9(0.8, 0.7, 1.0), kT=1e-4, u0=(0.02, 0.01), seed=r, stream=r,
                      init_mode=1, fields=f)
            for r, (nx, ny, f) in enumerate([(64, 64, (0, 9, 10)), (512, 32, (0,)), (16, 512, tuple(range(11))),
                                             (256, 256, (0, 1, 2, 3)), (2, 16, (0, 5))])]
    batch = Sim(reps, precision=precision)
    batch.run(12, 4)
    for r, p in enumerate(reps):
        one = Sim(p, precision=precision)
        one.run(12, 4)
        for a in p["fields"]:
            for b in p["fields"]:
                assert np.array_equal(batch.correlator(r, a, b), one.correlator(0, a, b)), (r, a, b)
