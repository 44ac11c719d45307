"""Plain lattices at the limits of their sweep in words (k_words.cu): many
replicas, rows beyond a launch's limit, a buffer without the room.  Integer
work: bit-exact against the plain kernels."""

import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001800


def _pair(ianus, **kw):
    a, b = (ianus.Lattice(layout="i8", seed=SEED, series_capacity=8, **kw) for _ in range(2))
    b.set_resident(0)
    return a, b


def _words_used(ianus, lat):
    """Whether a sweep since the room was cleared wrote the words."""
    return bool(lat.buffer[lat._lib.ianus_required_bytes(C.byref(lat.cfg)):].any())


def _equal(a, b):
    assert np.array_equal(a.spins(), b.spins())
    for x, y in zip(a.series(), b.series()):
        assert (x is None and y is None) or np.array_equal(x, y)


@pytest.mark.parametrize("L,S,R,words", [(40, 8, 128, False), (16, 64, 128, False), (16, 64, 110, True)])
def test_many_replicas(ianus, L, S, R, words):
    a, b = _pair(ianus, dim=3, L=L, n_samples=S, n_replicas=R)
    a.buffer[a._lib.ianus_required_bytes(C.byref(a.cfg)):].zero_()
    for algo, n, every in (("heatbath", 2, 0), ("metropolis", 4, 1), ("heatbath", 12, 5)):
        for lat in (a, b):
            lat.sweep(algo, 0.8, n, every)
    assert _words_used(ianus, a) == words
    _equal(a, b)


@pytest.mark.parametrize("R,words", [(17, False), (16, True), (2, True)])
def test_many_rows(ianus, R, words):
    a, b = _pair(ianus, dim=3, L=4, n_samples=64 * 4095, n_replicas=R)
    a.buffer[a._lib.ianus_required_bytes(C.byref(a.cfg)):].zero_()
    for lat in (a, b):
        lat.sweep("heatbath", 0.8, 6, 3)
    assert _words_used(ianus, a) == words
    _equal(a, b)


def test_couplings_written_in_the_buffer(ianus):
    """Spins and couplings changed in place, without a call, between two runs."""
    import torch

    a, b = _pair(ianus, dim=3, L=32, n_samples=70, n_replicas=2)
    nspins, ncouplings = 70 * 2 * 32 ** 3, 70 * 3 * 32 ** 3
    at = (nspins + 255) // 256 * 256
    gen = torch.Generator(device="cuda").manual_seed(5)
    a.buffer[a._lib.ianus_required_bytes(C.byref(a.cfg)):].zero_()
    for run in range(3):
        signs = torch.randint(0, 2, (ncouplings,), generator=gen, device="cuda", dtype=torch.int8) * 2 - 1
        flips = torch.randint(0, 2, (nspins,), generator=gen, device="cuda", dtype=torch.int8) * 2 - 1
        for lat in (a, b):
            lat.sweep("heatbath", 0.9, 20, 5)
            lat.buffer[at:at + ncouplings].view(torch.int8).mul_(signs)
            lat.buffer[:nspins].view(torch.int8).mul_(flips)
    for lat in (a, b):
        lat.sweep("heatbath", 0.9, 20, 5)
    assert _words_used(ianus, a)
    assert np.array_equal(a.couplings(), b.couplings())
    _equal(a, b)


def test_threads_with_different_replicas(ianus):
    """Two threads whose word sweeps ask for different amounts of shared memory."""
    import threading

    import torch

    pairs, failed = [], []
    for R in (108, 28):
        with torch.cuda.stream(torch.cuda.Stream()):
            pairs.append(_pair(ianus, dim=3, L=8, n_samples=200, n_replicas=R))

    def run(lat):
        try:
            for _ in range(60):
                lat.sweep("metropolis", 0.8, 20)
        except Exception as e:
            failed.append(e)

    for a, _ in pairs:
        a.set_graphs(False)
        a.buffer[a._lib.ianus_required_bytes(C.byref(a.cfg)):].zero_()
    torch.cuda.synchronize()
    threads = [threading.Thread(target=run, args=(a,)) for a, _ in pairs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for a, b in pairs:
        run(b)
        assert _words_used(ianus, a)
        _equal(a, b)


@pytest.mark.parametrize("short", [0, 1])
def test_a_buffer_without_room_for_the_words(ianus, short):
    """The least buffer, and one byte less than the preferred, sweep by bytes."""
    import torch

    a, b = _pair(ianus, dim=3, L=32, n_samples=70, n_replicas=2)
    lib = a._lib
    cfg = type(a.cfg)()
    C.memmove(C.byref(cfg), C.byref(a.cfg), C.sizeof(cfg))
    least, most = lib.ianus_required_bytes(C.byref(cfg)), lib.ianus_preferred_bytes(C.byref(cfg))
    size = most - 1 if short else least
    buf = torch.zeros(size, dtype=torch.uint8, device="cuda")
    cfg.device_buffer, cfg.device_buffer_bytes = buf.data_ptr(), size
    h = C.c_void_p()
    assert lib.ianus_lattice_create(C.byref(cfg), C.byref(h)) == 0
    beta = (C.c_double * 1)(0.9)
    assert lib.ianus_sweep(h, 1, beta, 30, 0) == 0
    b.sweep("heatbath", 0.9, 30)
    out = np.empty(b.spins().shape, dtype=np.int8)
    assert lib.ianus_get_spins_i8(h, out.ctypes.data) == 0
    assert np.array_equal(out, b.spins()) and not buf[least:].any()
    lib.ianus_destroy(h)
