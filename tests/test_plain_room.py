"""Which plain lattices ask for room for their words (host arithmetic of
ianus_preferred_bytes; no GPU needed)."""

import ctypes as C

import paper_0704_3573_gb300 as ianus


def _words_room(L, S, R, dim=3):
    c = ianus.IanusConfig()
    c.abi_version, c.dim, c.L, c.n_samples, c.n_replicas, c.n_temps = ianus.ABI_VERSION, dim, L, S, R, 1
    c.layout, c.occupation, c.seed, c.series_capacity = ianus._LAYOUTS["i8"], 1.0, 1, 2
    lib = ianus.lib()
    least, most = lib.ianus_required_bytes(C.byref(c)), lib.ianus_preferred_bytes(C.byref(c))
    assert 0 < least <= most
    return most - least


def test_no_words_beyond_the_replicas_their_sweep_takes():
    """The word sweep keeps 2112 bytes of threshold planes a replica in shared
    memory: 110 replicas fit 227 KiB."""
    assert _words_room(40, 8, 110) >= 8 * 110 * 40 ** 3
    assert _words_room(40, 8, 111) == 0
    assert _words_room(16, 64, 128) == 0
    assert _words_room(16, 64, 4000) == 0


def test_no_words_beyond_the_rows_their_measurement_takes():
    """The counts of three replicas and more are launched with a row of blocks
    per (group, replica), 65535 at most; one or two replicas are a row a group."""
    assert _words_room(4, 64 * 4095, 16) > 0
    assert _words_room(4, 64 * 4095, 17) == 0
    assert _words_room(4, 64 * 4095, 2) > 0
