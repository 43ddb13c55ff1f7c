"""FP64 D1Q3 runs at the limits of their chunked form (csrc/lb_d1q3_runs.cu), against the per-step
launches (GPU).  The arithmetic of a site is the same on both paths, so states are equal bit for bit."""
import numpy as np
import pytest

from paper_1010_1233_gb300 import Sim, workloads as W

pytestmark = pytest.mark.gpu


def _replica(nx, fields=(), **kw):
    args = dict(kT=1e-3, u0=(0.05, 0.0), seed=nx, init_mode=1)
    return W.replica("D1Q3", nx, 1, W.taus_d1q3(0.7), fields=fields, **{**args, **kw})


def _launches(sim, n, every):
    n0 = sim.kernel_launches()
    sim.run(n, every)
    return sim.kernel_launches() - n0


@pytest.mark.parametrize("sizes", [(4096,), (4098,), (4200,), (4266,), (4268,), (64, 4098), (64, 4266), (4096, 64)])
def test_lattices_wider_than_a_block_covers(sizes):
    # 1024 threads of four sites each take 4096 sites; wider lattices, and batches with one, run
    # one launch per step
    reps = [_replica(nx, stream=i) for i, nx in enumerate(sizes)]
    a, b = Sim(reps, precision="fp64"), Sim(reps, precision="fp64")
    b.set_graphs(False)
    for n in (3, 9):
        launched = _launches(a, n, 0)
        assert (launched < n) == (max(sizes) <= 4096), launched
        b.run(n)
    for r in range(len(reps)):
        assert np.array_equal(a.populations(r), b.populations(r)), r


@pytest.mark.parametrize("nx,fields", [(2, (0,)), (2, (0, 9)), (2, (0, 1, 2, 9)), (4, (1,)), (4, (0, 1)), (4, (0, 1, 2, 9)),
                                       (8, (2,)), (8, (0, 1)), (8, (0, 1, 2, 9)), (16, (0, 1, 2)), (2048, (0, 1, 2, 9))])
def test_sampled_lattices_of_every_size_run_in_chunks(nx, fields):
    # alone, and as the smallest of a batch, whose launches are sized by the largest of its replicas
    for reps in ([_replica(nx, fields)], [_replica(64, (0, 1, 2), stream=1), _replica(nx, fields), _replica(32, stream=2)]):
        a, b = Sim(reps, precision="fp64"), Sim(reps, precision="fp64")
        b.set_graphs(False)
        assert _launches(a, 45, 2) <= 4 * 12                    # a few launches a chunk; per step 45 + 2 x 23
        b.run(45, 2)
        for r, p in enumerate(reps):
            assert np.array_equal(a.populations(r), b.populations(r)), r
            for i, x in enumerate(p["fields"]):
                for y in p["fields"][i:]:
                    ca, na = a.correlator(r, x, y, with_count=True)
                    cb, nb = b.correlator(r, x, y, with_count=True)
                    # 23 samples in another order: 23 roundings of 2^-53 of the sum's size, and those of
                    # the transforms
                    assert na == nb == 23 and np.abs(ca - cb).max() <= 1e-13 * max(1.0, np.abs(cb).max()), (r, x, y)


def _sums(sim, reps, r=0):
    f = reps[r]["fields"]
    return [sim.correlator(r, x, y) for i, x in enumerate(f) for y in f[i:]]


@pytest.mark.parametrize("nx,fields", [(4, (0, 1)), (64, (0, 1, 2)), (64, (0, 1, 2, 9)), (1024, (1, 9))])
@pytest.mark.parametrize("every", [1, 7])
def test_sums_do_not_depend_on_calls_chunks_or_batch(nx, fields, every):
    # a sum takes one product per sample in the order of the steps, whatever the launches: equal bit
    # for bit for one call over several chunks (of at most 1024 steps), calls that end inside chunks and
    # sampling periods, one step a call, per-step launches, and in a batch
    p = _replica(nx, fields)
    others = [_replica(128, (0, 2), stream=2), _replica(30, stream=3)]
    n = 2100
    a = Sim([p], precision="fp64")
    assert 2 * 4 < _launches(a, n, every) < n                      # the chunked path, three chunks or more
    ref, pop = _sums(a, [p]), a.populations()

    def check(reps, runs, r=0, graphs=True):
        s = Sim(reps, precision="fp64")
        s.set_graphs(graphs)
        for k in runs:
            s.run(k, every)
        assert np.array_equal(s.populations(r), pop)
        for x, y in zip(_sums(s, reps, r), ref):
            assert np.array_equal(x, y)
        s.close()

    check([p], (n // 2, n - n // 2))
    check([p], (1,) * 40 + (n - 40,))
    check([p], (n,), graphs=False)
    check(others + [p], (5, 1030, n - 1035), r=2)


@pytest.mark.parametrize("sizes,every", [((1024,) * 310, 1), ((2048, 64, 4096, 30, 1024) * 70, 3), ((256,) * 700, 50),
                                         ((512,) * 400, 0), ((4096, 4096, 4096, 4096) * 76 + (8,) * 9, 1)])
def test_large_batches_run_in_groups_through_one_scratch(sizes, every):
    # batches of several groups of replicas (of 304 and 81,920 sites or more), the last group small, whose
    # chunks are shorter than the run (at most 256 MB of scratch); against single replicas, bit for bit
    reps = [_replica(nx, () if nx == 30 else (0, 2)[: 1 + i % 2], seed=7, stream=i, init_mode=0, kT=1e-4)
            for i, nx in enumerate(sizes)]
    n = 150
    sim = Sim(reps, precision="fp64")
    assert _launches(sim, n, every) > 2 * 2
    assert sim.workspace_bytes < 270e6 + 8000 * len(reps) + sum(sizes) * 8 * (6 + 2 + 8)   # state, fields, spectra, sums
    for r in sorted({0, 1, 3, len(reps) // 2, len(reps) // 2 + 1, len(reps) - 2, len(reps) - 1}):
        one = Sim(reps[r], precision="fp64")
        one.run(n, every)
        assert np.array_equal(sim.populations(r), one.populations()), r
        if every and reps[r]["fields"]:
            for x, y in zip(_sums(sim, reps, r), _sums(one, [reps[r]])):
                assert np.array_equal(x, y), r
        one.close()


def test_more_replicas_than_a_grid_dimension():
    # 65,535 blocks is the limit of a grid in y and z, 2^31 - 1 in x
    n, pick = 65_540, (0, 65_534, 65_535, 65_536, 65_539)
    reps = [_replica(16, fields=(0,), seed=5, stream=i, init_mode=0, u0=(0.01 * (i % 7), 0.0)) for i in range(n)]
    sim = Sim(reps, precision="fp64")
    assert _launches(sim, 9, 3) > 0
    sim.sync()
    for r in pick:
        one = Sim(reps[r], precision="fp64")
        one.set_graphs(False)
        one.run(9, 3)
        assert np.array_equal(sim.populations(r), one.populations()), r
        c, k = sim.correlator(r, 0, 0, with_count=True)
        c1, k1 = one.correlator(0, 0, 0, with_count=True)
        # three samples, added in another order: 2 roundings of 2^-53, and those of the transforms
        assert k == k1 == 3 and np.abs(c - c1).max() <= 1e-13 * max(1.0, np.abs(c1).max()), r
