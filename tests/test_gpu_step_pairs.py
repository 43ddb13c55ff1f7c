"""The FP32 D2Q9 step kernel for two and four sites per thread against the one-site kernel (GPU):
bit-identical states and sampled fields at the edges of its units and blocks -- rows of two
sites, one row, rows that end inside a warp, lattices of less than a block and of blocks of a
quarter, every noise mode, masks without noise, uneven batches whose blocks change replica; and
the FP64 steps that are launched early against plain launches."""
import numpy as np
import pytest

from paper_1010_1233_gb300 import Sim, workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(2, 1), (2, 9), (4, 4), (6, 5), (36, 11), (64, 64), (130, 33), (516, 7), (1030, 64), (256, 900)]


def _states(reps, vec, every):
    sim = Sim(reps)
    sim.set_step_config(vec)
    sim.run(7, every)
    out = [sim.populations(r) for r in range(len(reps))]
    if every:
        out += [sim.fields(r) for r in range(len(reps))]
    return out


@pytest.mark.parametrize("mode,mask", [(0, None), (1, None), (2, None), (0, 0), (0, 0b000111000)])
def test_pairs_equal_single_sites(mode, mask):
    for nx, ny in SHAPES:
        p = W.replica("D2Q9", nx, ny, W.taus_d2q9(0.6, 0.8, 1.1), kT=1e-3, u0=(0.1, -0.05), seed=nx + ny, init_mode=1,
                      noise_mode=mode, noise_mask=mask)
        one = _states([p], 1, 0)
        for vec in (2, 4):
            if nx % vec == 0:
                assert np.array_equal(_states([p], vec, 0)[0], one[0]), (nx, ny, vec)


@pytest.mark.parametrize("fields", [(0,), (3, 9), tuple(range(11))])
def test_batched_pairs_and_fields(fields):
    shapes = [(64, 64), (4, 2), (512, 32), (16, 16), (256, 128)]
    reps = [W.replica("D2Q9", nx, ny, W.taus_d2q9(0.7, 0.8, 1.0), kT=1e-3, u0=(0.02 * r, 0.01), seed=r, stream=r,
                      init_mode=1, fields=fields, noise_mode=r % 3) for r, (nx, ny) in enumerate(shapes)]
    one = _states(reps, 1, 3)
    for vec in (2, 4):
        for a, b in zip(_states(reps, vec, 3), one):
            assert np.array_equal(a, b), vec


@pytest.mark.parametrize("lat,dims", [("D2Q9", (2, 1)), ("D2Q9", (16, 16)), ("D2Q9", (254, 67)), ("D2Q9", (256, 266)),
                                      ("D2Q9", (320, 256)), ("D3Q15", (6, 5, 4)), ("D3Q15", (48, 32, 25)),
                                      ("D3Q15", (64, 48, 40)), ("D3Q19", (32, 19, 64))])
def test_early_launches_equal_plain_ones(lat, dims):
    # FP64 steps launched beside the step before (one unit per thread) against one block that loops
    # over everything, launched after it: the same states, sampled or not, in and out of graphs
    kw = dict(kT=1e-3, seed=sum(dims), init_mode=1, fields=(0, 4))
    p = (W.replica("D2Q9", *dims, W.taus_d2q9(0.6, 0.8, 1.1), u0=(0.1, -0.05), **kw) if lat == "D2Q9" else
         W.replica3(*dims, (W.taus_d3q15 if lat == "D3Q15" else W.taus_d3q19)(0.7, 0.9, 1.1), u0=(0.05, -0.02, 0.03),
                    lattice=lat, **kw))
    pow2 = lat != "D2Q9" or all(n & (n - 1) == 0 for n in dims)
    every = 5 if pow2 else 0
    if not pow2:
        p["fields"] = ()
    a, b = Sim(p, precision="fp64"), Sim(p, precision="fp64")
    b.set_step_config(1, 1)
    for n in (3, 70, 9):
        a.run(n, every)
        b.run(n, every)
    assert np.array_equal(a.populations(), b.populations())
    if every:
        assert np.array_equal(a.fields(), b.fields())
