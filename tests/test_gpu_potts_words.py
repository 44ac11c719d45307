"""GPU parity of the Potts word kernels (4 samples worked on together) where
they can go wrong: one or two replicas a thread (odd and even replica
counts), one temperature (rows in shared memory) or several, samples that
leave a word part-filled, L = 2 (one word per row and colour), sides whose
colour half is no multiple of a warp, blocks that span several quads, and
counts at both ends (ferromagnet and beta = 0).  Integer work: bit-exact."""

import numpy as np
import pytest

import oracle as orc_mod
from oracle import HEATBATH, Oracle

pytestmark = pytest.mark.gpu

SEED = 0x0704357300000B00
MODELS = {"potts": orc_mod.MODEL_POTTS, "potts_perm": orc_mod.MODEL_PERM}
CASES = [(3, 2, 5, 2, 1), (3, 6, 3, 1, 1), (3, 6, 9, 4, 1), (3, 8, 4, 2, 2), (3, 4, 6, 3, 3), (2, 2, 1, 2, 1),
         (2, 10, 7, 2, 1), (2, 34, 5, 3, 1), (3, 20, 2, 2, 1)]


@pytest.mark.parametrize("ferro", [False, True])
@pytest.mark.parametrize("model,dim,L,S,R,K", [(m, *c) for m in MODELS for c in CASES] +
                         [("potts_perm", 4, 2, 3, 2, 1), ("potts_perm", 4, 6, 5, 1, 1), ("potts_perm", 4, 4, 2, 4, 2)])
def test_potts_words_match_oracle(ianus, model, dim, L, S, R, K, ferro):
    beta = [1.1, 0.0, 2.0][:K]
    lat = ianus.Lattice(model=model, dim=dim, L=L, n_samples=S, n_replicas=R, n_temps=K, seed=SEED + L, ferro=ferro)
    orc = Oracle(model=MODELS[model], dim=dim, L=L, sample_ids=list(range(S)), n_replicas=R, n_temps=K, seed=SEED + L,
                 disorder=orc_mod.DIS_FERRO if ferro else orc_mod.DIS_EA)
    if ferro and model == "potts_perm":  # identity permutations, which the oracle takes as given couplings
        orc.set_couplings(lat.couplings())
    for n in (1, 2, 5):
        lat.sweep(HEATBATH, beta, n, measure_every=1)
        orc.sweep(HEATBATH, beta, n, measure_every=1)
    assert np.array_equal(lat.spins(), orc.spins())
    _, E, M, Q = lat.series()
    _, Eo, Mo, Qo = orc.series()
    assert np.array_equal(E, Eo) and np.array_equal(M, Mo)
    if R >= 2:
        assert np.array_equal(Q, Qo)
