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
