"""Plain lattices of many samples swept in words (k_words.cu): part-filled
groups, sides that are no power of two, measurements, new temperatures,
couplings and states set between runs, and a buffer without room for the words.
Integer work: bit-exact against the plain kernels."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001600


@pytest.mark.parametrize("dim,L,S,R", [(3, 32, 64, 1), (3, 34, 70, 2), (3, 22, 200, 3), (2, 130, 129, 2), (3, 40, 17, 1),
                                       (2, 64, 250, 4), (3, 64, 9, 3)])
def test_words_equal_plain_kernels(ianus, dim, L, S, R):
    a, b = (ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, seed=SEED + L, layout="i8", series_capacity=12)
            for _ in range(2))
    b.set_resident(0)
    rng = np.random.default_rng(L)
    for algo, beta, n, every in (("heatbath", 0.9, 20, 0), ("metropolis", 0.7, 20, 4), ("metropolis", 0.7, 21, 7),
                                 ("heatbath", 0.9, 40, 1)):
        for lat in (a, b):
            lat.sweep(algo, beta, n, every)
        for x, y in zip(a.measure(), b.measure()):
            assert (x is None and y is None) or np.array_equal(x, y)
        if every == 7:
            J = rng.choice(np.array([-1, 1], dtype=np.int8), size=a.couplings().shape)
            state = b.get_state()
            for lat in (a, b):
                lat.set_couplings(J)
        if every == 0:
            spins = rng.choice(np.array([-1, 1], dtype=np.int8), size=a.spins().shape)
            for lat in (a, b):
                lat.set_spins(spins)
    assert np.array_equal(a.spins(), b.spins())
    for x, y in zip(a.series(), b.series()):
        assert (x is None and y is None) or np.array_equal(x, y)
    for lat in (a, b):  # back to the earlier couplings, spins and counters
        lat.set_state(state)
        lat.sweep("heatbath", 0.9, 24, 5)
    assert np.array_equal(a.spins(), b.spins())
