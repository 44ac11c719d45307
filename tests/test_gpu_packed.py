"""Resident sweeps of small plain lattices with 32 sites a word (k_packed.cu):
whole-row words and unaligned ones, one word to a thousand, samples that share
a group's random numbers, runs longer than the decisions that are kept at a
time, series rings that wrap, and a buffer without room for the decisions.
Integer work: bit-exact."""

import ctypes as C

import numpy as np
import pytest

from oracle import HEATBATH, METROPOLIS, Oracle

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001400


@pytest.mark.parametrize("algo,beta", [(METROPOLIS, 0.7), (HEATBATH, 1.1), (METROPOLIS, 0.0), (HEATBATH, 50.0)])
@pytest.mark.parametrize("dim,L,S,R", [(3, 4, 1, 1), (3, 8, 3, 2), (3, 12, 65, 1), (2, 8, 2, 1), (2, 24, 3, 1),
                                       (2, 64, 1, 2), (3, 16, 1, 1)])
def test_packed_equals_oracle(ianus, dim, L, S, R, algo, beta):
    lat = ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, seed=SEED + L, layout="i8", series_capacity=7)
    orc = Oracle(dim=dim, L=L, sample_ids=list(range(S)), n_replicas=R, seed=SEED + L)
    for n, every in ((13, 2), (9, 1)) if R == 1 else ((13, 0), (9, 0)):
        lat.sweep(algo, beta, n, every)
        orc.sweep(algo, beta, n, every)
    assert np.array_equal(lat.spins(), orc.spins())
    if R == 1:
        sweep, E, M, _ = lat.series()
        so, Eo, Mo, _ = orc.series()
        assert np.array_equal(E, Eo[-7:]) and np.array_equal(M, Mo[-7:]) and list(sweep) == list(so)[-7:]


@pytest.mark.parametrize("dim,L,S,R,n", [(3, 36, 1, 1, 40), (2, 256, 2, 1, 40), (3, 16, 100, 1, 70), (3, 8, 70, 3, 300),
                                         (3, 20, 30, 2, 90), (2, 120, 5, 1, 50)])
def test_packed_equals_launched(ianus, dim, L, S, R, n):
    a, b = (ianus.Lattice(dim=dim, L=L, n_samples=S, n_replicas=R, seed=SEED, layout="i8", series_capacity=200)
            for _ in range(2))
    b.set_resident(0)
    every = 1 if R == 1 else 0
    for lat in (a, b):
        lat.sweep("heatbath", 0.8, n, every)
        lat.sweep("metropolis", 0.9, n, 3 * every)
    assert np.array_equal(a.spins(), b.spins())
    if every:
        for x, y in zip(a.series(), b.series()):
            assert (x is None and y is None) or np.array_equal(x, y)


def test_a_smaller_buffer_sweeps_without_the_decisions(ianus):
    import torch
    a = ianus.Lattice(dim=3, L=8, n_samples=2, seed=SEED, layout="i8")
    lib = a._lib
    cfg = type(a.cfg)()
    C.memmove(C.byref(cfg), C.byref(a.cfg), C.sizeof(cfg))
    least = lib.ianus_required_bytes(C.byref(cfg))
    assert cfg.device_buffer_bytes == lib.ianus_preferred_bytes(C.byref(cfg)) == least + 1024 * 2 * 512
    buf = torch.empty(least, dtype=torch.uint8, device="cuda")
    cfg.device_buffer, cfg.device_buffer_bytes = buf.data_ptr(), least
    h = C.c_void_p()
    assert lib.ianus_lattice_create(C.byref(cfg), C.byref(h)) == 0
    beta = (C.c_double * 1)(0.9)
    assert lib.ianus_sweep(h, HEATBATH, beta, 30, 0) == 0
    a.sweep("heatbath", 0.9, 30)
    out = np.empty(a.spins().shape, dtype=np.int8)
    assert lib.ianus_get_spins_i8(h, out.ctypes.data) == 0
    assert np.array_equal(out, a.spins())
    lib.ianus_destroy(h)
    cfg.device_buffer_bytes = least - 1
    assert lib.ianus_lattice_create(C.byref(cfg), C.byref(h)) != 0
