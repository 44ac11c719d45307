"""Captured blocks of sweeps with their measurements (and several chains of
launches in one block): the same spins, series and exchanges as launch by
launch, over calls that end inside a block, cadences that change, a series
ring that wraps, lattices of one and of several chains, and every layout."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001100
LATTICES = [dict(dim=3, L=10, n_samples=70, n_replicas=2),
            dict(dim=2, L=12, n_samples=3, n_replicas=3),
            dict(dim=3, L=6, n_samples=65, n_replicas=2, n_temps=3),
            dict(dim=3, L=12, n_samples=10, n_replicas=2, disorder="rfim", field=1.0),
            dict(dim=3, L=34, n_samples=5, n_replicas=2, layout="i8"),
            dict(dim=2, L=10, n_samples=3, n_replicas=2, rng="wheel"),
            dict(model="potts", dim=3, L=8, n_samples=9, n_replicas=2),
            dict(model="potts_perm", dim=2, L=8, n_samples=5, n_replicas=3),
            # several chains
            dict(dim=3, L=40, n_samples=130, n_replicas=2),
            dict(dim=3, L=30, n_samples=156, n_replicas=1, disorder="daff", field=0.6, occupation=0.7),
            dict(dim=3, L=32, n_samples=64, n_replicas=3, n_temps=3),
            dict(dim=3, L=32, n_samples=130, n_replicas=1, layout="i8"),
            dict(model="potts", dim=3, L=24, n_samples=40, n_replicas=2)]
CALLS = [(5, 2), (64, 1), (64, 1), (7, 7), (30, 3), (33, 3), (33, 3), (9, 0), (11, 1)]


@pytest.mark.parametrize("kw", LATTICES, ids=lambda kw: "-".join(str(v) for v in kw.values()))
def test_measured_blocks_equal_launches(ianus, kw):
    a, b = (ianus.Lattice(seed=SEED, series_capacity=40, **kw) for _ in range(2))
    b.set_graphs(False)
    beta = [1.1, 0.8, 0.5][:a.K] if a.K > 1 else 1.0
    for n, every in CALLS:
        for lat in (a, b):
            lat.sweep("heatbath", beta, n, every)
            if a.K > 1 and n % 2 == 0 and not kw.get("disorder"):
                lat.pt_swap()
        if n != 64:
            continue
        for x, y in zip(a.series(), b.series()):
            assert (x is None) == (y is None) and (x is None or np.array_equal(x, y))
    assert a.sweeps == b.sweeps
    for x, y in zip(a.series(), b.series()):
        assert (x is None) == (y is None) and (x is None or np.array_equal(x, y))
    assert np.array_equal(a.spins(), b.spins())
    if a.K > 1:
        assert all(np.array_equal(x, y) for x, y in zip(a.pt_state()[:2], b.pt_state()[:2]))


@pytest.mark.parametrize("layout", ["bits64", "i8"])
@pytest.mark.parametrize("L,S,R,K,every", [(6, 5, 2, 4, 1), (8, 70, 1, 3, 2), (32, 70, 2, 4, 5), (12, 3, 3, 33, 3)])
def test_tempering_blocks_equal_calls(ianus, L, S, R, K, every, layout):
    if layout == "i8" and S * L > 1000:
        S = 3
    beta = [1.3 - 0.9 * k / K for k in range(K)]
    a, b = (ianus.Lattice(dim=3, L=L, n_samples=S, n_replicas=R, n_temps=K, seed=SEED, layout=layout,
                          series_capacity=60) for _ in range(2))
    b.set_graphs(False)
    for n, m in ((8, every), (24, every), (24, every), (24, 0), (24, 0), (7, 1), (24, every)):
        a.sweep_pt("metropolis", beta, n * every, every, m)
        for _ in range(n):
            b.sweep("metropolis", beta, every, m)
            b.pt_swap()
    for x, y in zip(a.series(), b.series()):
        assert (x is None) == (y is None) and (x is None or np.array_equal(x, y))
    assert np.array_equal(a.spins(), b.spins())
    assert all(np.array_equal(x, y) for x, y in zip(a.pt_state()[:2], b.pt_state()[:2]))
    assert a.pt_state()[2] == b.pt_state()[2]
