"""GPU parity of the lane-queue kernel's forms beside the one-temperature EA
sweep: random fields and dilution (tables per sign of s h, four class planes),
and per-lane threshold planes (several temperatures, more than two replicas).
Sizes where the split can go wrong: L = 2, sides that are no power of two,
part-filled words, one and two replicas a thread, blocks with fewer words than
threads, temperatures that queue many lanes or none.  Integer work: bit-exact."""

import numpy as np
import pytest

from oracle import DIS_DAFF, DIS_RFIM, HEATBATH, METROPOLIS, Oracle

pytestmark = pytest.mark.gpu

SEED = 0x0704357300000F00
NAMES = {DIS_RFIM: "rfim", DIS_DAFF: "daff"}


def _same(lat, orc, algo, beta):
    for n in (1, 4):
        lat.sweep(algo, beta, n, measure_every=2)
        orc.sweep(algo, beta, n, measure_every=2)
    assert np.array_equal(lat.spins(), orc.spins())
    _, E, M, Q = lat.series()
    _, Eo, Mo, Qo = orc.series()
    assert np.array_equal(E, Eo) and np.array_equal(M, Mo)
    if lat.R >= 2:
        assert np.array_equal(Q, Qo)


@pytest.mark.parametrize("beta", [0.0, 0.7, 30.0])
@pytest.mark.parametrize("algo", [METROPOLIS, HEATBATH])
@pytest.mark.parametrize("disorder,h,occ", [(DIS_RFIM, 1.25, 1.0), (DIS_RFIM, 9.0, 1.0), (DIS_DAFF, 0.75, 0.6),
                                            (DIS_DAFF, 1.5, 0.0)])
@pytest.mark.parametrize("dim,L,S,R", [(3, 2, 3, 1), (3, 10, 70, 2), (2, 6, 65, 2), (2, 12, 3, 1)])
def test_field_forms_match_oracle(ianus, dim, L, S, R, disorder, h, occ, algo, beta):
    lat = ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, seed=SEED + L, layout="bits64",
                        disorder=NAMES[disorder], field=h, occupation=occ)
    lat.set_variant(24)  # the lane-queue kernel at any size
    _same(lat, Oracle(dim=dim, L=L, sample_ids=list(range(S)), n_replicas=R, seed=SEED + L, disorder=disorder,
                      field=h, occupation=occ), algo, beta)


@pytest.mark.parametrize("algo", [METROPOLIS, HEATBATH])
@pytest.mark.parametrize("dim,L,S,R,K", [(3, 2, 1, 1, 3), (3, 10, 66, 3, 1), (3, 8, 5, 4, 2), (2, 6, 130, 1, 4),
                                         (2, 34, 3, 6, 1), (3, 14, 64, 2, 2)])
def test_lane_forms_match_oracle(ianus, dim, L, S, R, K, algo):
    beta = [1.2, 40.0, 0.3, 0.0][:K]
    lat = ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, n_temps=K, seed=SEED + L, layout="bits64")
    _same(lat, Oracle(dim=dim, L=L, sample_ids=list(range(S)), n_replicas=R, n_temps=K, seed=SEED + L), algo, beta)
