"""Chunked FP64 D1Q3 runs (csrc/lb_d1q3_runs.cu) at the edges of their split (GPU): lattices that do
not fill a warp, wider than a block (several sites per thread), runs across chunk ends and sampling
periods that do not divide them, every noise form, uneven batches with replicas that sample nothing;
against the per-step launches, which do the same arithmetic (states equal bit for bit; the sums
are added in another order: 1e-13 of their size), and short runs against the FP64 oracle."""
import numpy as np
import pytest

from oracle import lb
from paper_1010_1233_gb300 import Sim, workloads as W

pytestmark = pytest.mark.gpu


def _pair(reps, runs, every):
    a, b = Sim(reps, precision="fp64"), Sim(reps, precision="fp64")
    b.set_graphs(False)
    for n in runs:
        a.run(n, every)
        b.run(n, every)
    for r, p in enumerate(reps):
        assert np.array_equal(a.populations(r), b.populations(r)), r
        fl = list(p["fields"])
        if every and fl:
            assert np.array_equal(a.fields(r), b.fields(r)), r
        for i, x in enumerate(fl if every else []):
            for y in fl[i:]:
                ca, na = a.correlator(r, x, y, with_count=True)
                cb, nb = b.correlator(r, x, y, with_count=True)
                assert na == nb
                assert np.abs(ca - cb).max() <= 1e-13 * max(1.0, np.abs(cb).max()), (r, x, y)


@pytest.mark.parametrize("nx,fields", [(2, (0,)), (8, (0, 1)), (32, (0, 1, 2)), (64, (0, 1)), (1024, (0, 9)),
                                       (2048, (1,)), (30, ()), (1100, ())])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_runs_match_steps(nx, fields, mode):
    p = W.replica("D1Q3", nx, 1, W.taus_d1q3(0.7), kT=1e-3, u0=(0.05, 0.0), seed=nx, init_mode=1, fields=fields,
                  noise_mode=mode)
    _pair([p], (3, 1, 37), 3 if fields else 0)


def test_chunk_ends_and_uneven_batch():
    reps = [W.replica("D1Q3", 64, 1, W.taus_d1q3(0.8), kT=1e-4, seed=1, init_mode=1, fields=(0, 1, 2, 9)),
            W.replica("D1Q3", 16, 1, W.taus_d1q3(0.6), kT=1e-4, seed=2, stream=1, init_mode=1),
            W.replica("D1Q3", 4, 1, W.taus_d1q3(0.9), kT=1e-4, seed=3, stream=2, init_mode=1, fields=(2,), noise_mask=0),
            W.replica("D1Q3", 256, 1, W.taus_d1q3(0.9), kT=1e-4, seed=4, stream=3, init_mode=1, fields=(0, 1))]
    for every in (1, 7, 1500):
        _pair(reps, (1025, 2050), every)


def test_run_matches_oracle():
    p = W.replica("D1Q3", 40, 1, W.taus_d1q3(0.55), kT=1e-3, u0=(0.2, 0.0), seed=9, init_mode=1)
    sim, ref = Sim(p, precision="fp64"), lb.Run(lb.Params(**p))
    sim.run(60)
    ref.run(60)
    dev = np.abs(ref.f - lb.uniform_state(ref.p)).max()
    assert np.abs(sim.populations() - ref.f).max() < 60 * 1e-13 * dev      # ~10 roundings of 2^-53 f / dev a step
