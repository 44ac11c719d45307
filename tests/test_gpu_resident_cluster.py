"""Cluster-resident sweeps of small bit-sliced lattices against the oracle:
2D and 3D, L = 2 (fewer rows than blocks), sides whose rows do not divide
evenly among the blocks, part-filled words, several replicas and
temperatures, more words than threads, temperatures that decide every lane
late or at once, launches of many sweeps and captured blocks with
measurements.  Integer work: bit-exact."""

import numpy as np
import pytest

from oracle import HEATBATH, METROPOLIS, Oracle

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001200


@pytest.mark.parametrize("algo", [METROPOLIS, HEATBATH])
@pytest.mark.parametrize("dim,L,S,R,K", [(3, 2, 3, 1, 1), (3, 4, 65, 2, 1), (3, 6, 5, 3, 1), (3, 8, 64, 2, 2),
                                         (3, 10, 70, 1, 3), (2, 2, 1, 2, 1), (2, 10, 66, 2, 1), (2, 34, 3, 4, 1),
                                         (3, 16, 2, 4, 1), (3, 20, 1, 2, 1)])
def test_cluster_sweeps_match_oracle(ianus, dim, L, S, R, K, algo):
    beta = [0.9, 40.0, 0.0][:K]
    lat = ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, n_temps=K, seed=SEED + L, layout="bits64")
    lat.set_resident(3)  # a cluster wherever one can be formed
    orc = Oracle(dim=dim, L=L, sample_ids=list(range(S)), n_replicas=R, n_temps=K, seed=SEED + L)
    for n, every in ((1, 0), (2, 0), (9, 4), (12, 2), (12, 2)):
        lat.sweep(algo, beta, n, every)
        orc.sweep(algo, beta, n, measure_every=every)
    assert np.array_equal(lat.spins(), orc.spins())
    _, E, M, Q = lat.series()
    _, Eo, Mo, Qo = orc.series()
    assert np.array_equal(E, Eo) and np.array_equal(M, Mo)
    if R >= 2:
        assert np.array_equal(Q, Qo)


def test_cluster_sweeps_equal_launches(ianus):
    a, b = (ianus.Lattice(dim=3, L=12, n_samples=100, n_replicas=2, seed=SEED, layout="bits64") for _ in range(2))
    a.set_resident(3)
    b.set_resident(0)
    for n in (500, 3, 5000):
        a.sweep(HEATBATH, 1.0, n)
        b.sweep(HEATBATH, 1.0, n)
    assert np.array_equal(a.spins(), b.spins())
