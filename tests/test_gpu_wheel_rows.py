"""GPU parity of the wheel sweep and the plain measurement where their split
of the work changes: rows longer than one chunk of 32 sites a colour (and its
last, short chunk), rows whose count is no multiple of 4 or of a warp's rows,
sides that are and are not multiples of 4, warps of 4, 8 and 16 rows, and
measurements of one block and of several per configuration."""

import numpy as np
import pytest

from oracle import HEATBATH, METROPOLIS, RNG_WHEEL, Oracle

pytestmark = pytest.mark.gpu

SEED = 0x0704357300000E00


@pytest.mark.parametrize("algo", [METROPOLIS, HEATBATH])
@pytest.mark.parametrize("dim,L,S,R", [(2, 66, 2, 1), (2, 68, 1, 2), (2, 128, 3, 1), (2, 134, 2, 2), (3, 12, 2, 3),
                                       (3, 22, 3, 2), (3, 36, 1, 1), (2, 20, 700, 2), (2, 18, 1300, 1)])
def test_wheel_rows_match_oracle(ianus, dim, L, S, R, algo):
    ids = list(range(S)) if S < 8 else [0, 1, S // 2, S - 1]
    lat = ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, seed=SEED + L, layout="i8", rng="wheel")
    orc = Oracle(dim=dim, L=L, sample_ids=ids, n_replicas=R, seed=SEED + L, rng=RNG_WHEEL)
    for n in (1, 3):
        lat.sweep(algo, 0.8, n, measure_every=2)
        orc.sweep(algo, 0.8, n, measure_every=2)
    assert np.array_equal(lat.spins()[ids], orc.spins())
    _, E, M, Q = lat.series()
    _, Eo, Mo, Qo = orc.series()
    assert np.array_equal(E[:, ids], Eo) and np.array_equal(M[:, ids], Mo)
    if R >= 2:
        assert np.array_equal(Q[:, ids], Qo)
