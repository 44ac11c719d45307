"""Plain lattices of more than one 64-sample group whose sweeps are captured as
several chains: parallel tempering (each chain's sweeps after the swap step)
and measurements, over cadences and repeated calls.  Integer work: bit-exact
against launch by launch."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001700


def _equal(a, b):
    for x, y in zip(a.series(), b.series()):
        assert (x is None) == (y is None) and (x is None or np.array_equal(x, y))
    assert np.array_equal(a.spins(), b.spins())
    if a.K > 1:
        assert all(np.array_equal(x, y) for x, y in zip(a.pt_state()[:2], b.pt_state()[:2]))
        assert a.pt_state()[2] == b.pt_state()[2]


@pytest.mark.parametrize("dim,L,S,R,K", [(3, 32, 130, 2, 4), (2, 64, 130, 2, 4), (2, 32, 300, 1, 40), (3, 32, 70, 2, 2)])
@pytest.mark.parametrize("every", [1, 2, 5])
def test_tempering_in_chains_equals_calls(ianus, dim, L, S, R, K, every):
    beta = [1.3 - 0.9 * k / K for k in range(K)]
    a, b = (ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, n_temps=K, seed=SEED + L, layout="i8",
                          series_capacity=60) for _ in range(2))
    b.set_graphs(False)
    for n, m in ((24, every), (24, every), (24, 0), (24, 0), (7, every), (24, every)):
        a.sweep_pt("heatbath", beta, n * every, every, m)
        for _ in range(n):
            b.sweep("heatbath", beta, every, m)
            b.pt_swap()
    _equal(a, b)


@pytest.mark.parametrize("dim,L,S,R,K", [(3, 32, 200, 2, 1), (2, 128, 130, 1, 1), (3, 64, 129, 1, 2)])
def test_measured_chains_equal_launches(ianus, dim, L, S, R, K):
    beta = [0.9, 0.6][:K] if K > 1 else 0.9
    a, b = (ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, n_temps=K, seed=SEED + L, layout="i8",
                          series_capacity=60) for _ in range(2))
    b.set_graphs(False)
    for lat in (a, b):
        lat.set_resident(0)  # the byte kernels, also with one temperature
        for n, every in ((16, 2), (16, 2), (16, 2), (20, 5), (20, 5), (9, 1), (9, 1), (9, 1)):
            lat.sweep("metropolis", beta, n, every)
    _equal(a, b)
