"""GPU parity of the plain layout's kernels as they are chosen by size: the
thread-per-update kernel, the shared-plane kernels with 8 to 64 samples a
thread (word and byte form), and the resident sweep where it pays.  Sample
counts end inside a chunk of 8, at its end, and in a second group."""

import numpy as np
import pytest

from oracle import HEATBATH, METROPOLIS, Oracle

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001000


@pytest.mark.parametrize("resident", [1, 0])
@pytest.mark.parametrize("algo", [METROPOLIS, HEATBATH])
@pytest.mark.parametrize("dim,L,S,R", [(3, 12, 9, 2), (3, 12, 64, 1), (3, 10, 70, 2), (3, 10, 8, 1), (2, 22, 100, 1),
                                       (2, 36, 17, 2), (3, 34, 2, 1), (2, 160, 130, 1)])
def test_plain_kernels_match_oracle(ianus, dim, L, S, R, algo, resident):
    ids = list(range(S)) if S * L ** dim < 40000 else sorted({0, 1, S // 2, S - 1})
    lat = ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, seed=SEED + L, layout="i8")
    lat.set_resident(resident)  # 0: the shared-plane kernels at any size
    orc = Oracle(dim=dim, L=L, sample_ids=ids, n_replicas=R, seed=SEED + L)
    for n in (1, 4):
        lat.sweep(algo, 0.8, n, measure_every=2)
        orc.sweep(algo, 0.8, n, measure_every=2)
    assert np.array_equal(lat.spins()[ids], orc.spins())
    _, E, M, Q = lat.series()
    _, Eo, Mo, Qo = orc.series()
    assert np.array_equal(E[:, ids], Eo) and np.array_equal(M[:, ids], Mo)
    if R >= 2:
        assert np.array_equal(Q[:, ids], Qo)
