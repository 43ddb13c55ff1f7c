"""Tiles of the sampling passes on short and wide lattices (GPU): column transforms that take up to 1024
columns to a block, with columns past the last one; accumulation tiles left whole or cut; fewer row pairs
per block on launches of few rows.  Against numpy's FFT in FP64.

Tolerance: a transform of V points has a relative error of ~log2(V) roundings in the root mean square over
its points; products double it: 4 log2(V) eps of the largest sum."""
import numpy as np
import pytest
import torch

from paper_1010_1233_gb300 import Sim, workloads as W
from paper_1010_1233_gb300.sim import spectra_accumulate, unpack_pair_sums

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("F,ny,nx", [(1, 2, 8192), (2, 4, 4096), (9, 8, 2048), (4, 8, 4096), (3, 8, 1024), (9, 8, 64), (3, 32, 1024),
                                     (2, 512, 32), (1, 4096, 256), (3, 4096, 64), (1, 1, 1024), (3, 2, 512), (7, 16, 16),
                                     (11, 1024, 16)])
def test_pair_sums_of_short_and_wide_lattices(precision, F, ny, nx):
    dt, eps = (torch.float64, 2.0 ** -53) if precision == "fp64" else (torch.float32, 2.0 ** -24)
    x = torch.tensor(W.random_perturbation((F, ny, nx), F + ny + nx), dtype=dt, device="cuda")
    sums, mean0 = spectra_accumulate(x)
    k = np.fft.rfft2(x.double().cpu().numpy())
    tol = 4 * np.log2(nx * ny) * eps
    assert np.abs(mean0.cpu().numpy() - k[:, 0, 0].real).max() <= tol * np.abs(k).max()
    for (a, b), g in unpack_pair_sums(sums, F, ny, nx).items():
        scale = np.abs(k[a]).max() * np.abs(k[b]).max()
        assert np.abs(g - k[a] * k[b].conj()).max() <= tol * scale, (a, b)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_uneven_short_replicas_equal_single_runs(precision):
    # one-pass columns of 2 to 512 points, tiles of 4 to 512 columns, in one launch; a replica's sums are its own
    reps = [W.replica("D2Q9", nx, ny, W.taus_d2q9(0.8, 0.7, 1.0), kT=1e-4, u0=(0.02, 0.01), seed=r, stream=r,
                      init_mode=1, fields=f)
            for r, (nx, ny, f) in enumerate([(2048, 8, (0, 9, 10)), (2, 256, (0,)), (512, 2, tuple(range(11))),
                                             (64, 512, (0, 1, 2)), (256, 32, (0, 5)), (1024, 4, (9,))])]
    batch = Sim(reps, precision=precision)
    batch.run(12, 4)
    for r, p in enumerate(reps):
        one = Sim(p, precision=precision)
        one.run(12, 4)
        for i, a in enumerate(p["fields"]):
            for b in p["fields"][i:]:
                assert np.array_equal(batch.correlator(r, a, b), one.correlator(0, a, b)), (r, a, b)
