"""A pool's jobs against the same jobs on their own lattices, at the sizes
where the fused sweep gives a word four, two and one threads, with one job a
group and many, jobs that end inside a block of sweeps, and pools swept in
captured blocks and one sweep at a time."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HB, METRO = 1, 0


@pytest.mark.parametrize("dim,L,groups", [(3, 4, 1), (3, 10, 2), (2, 34, 1), (3, 32, 1), (2, 128, 4), (3, 40, 2)])
def test_pool_jobs_equal_their_own_lattices(ianus, dim, L, groups):
    jobs = [(0, 0, 64, HB, 0.8, 40)]  # group, first lane, samples, algorithm, beta, sweeps
    if groups > 1:
        jobs += [(1, 0, 1, METRO, 1.3, 7), (1, 1, 20, HB, 0.5, 100), (1, 40, 24, METRO, 40.0, 26)]
    pool = ianus.Lattice(dim=dim, L=L, n_samples=64 * groups, seed=1, layout="bits64", series_capacity=1)
    for k, (g, lane0, n, algo, beta, sweeps) in enumerate(jobs):
        pool.segment_load(g, lane0, n, 77 + k, algo, beta, sweeps)
    for n in (1, 20, 3, 12):
        pool.sweep_segments(n)
    spins = pool.spins()
    for k, (g, lane0, n, algo, beta, sweeps) in enumerate(jobs):
        own = ianus.Lattice(dim=dim, L=L, n_samples=n, seed=77 + k, layout="bits64", series_capacity=1)
        own.sweep(algo, beta, min(sweeps, 36))
        assert pool.segment_state(g, lane0) == (min(sweeps, 36), sweeps)
        lo = 64 * g + lane0
        assert np.array_equal(spins[lo:lo + n], own.spins())
        own.close()
