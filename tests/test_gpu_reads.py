"""Results read through page-locked memory and, when large, directly: several
arrays and threads at once, and arrays that are page-locked themselves."""

import ctypes as C
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x0704357300001500


# a few bytes, arrays below and above the staged size, more than a block in all, a ring that wraps
@pytest.mark.parametrize("S,K,R,rows", [(1, 1, 1, 1), (70, 3, 2, 9), (512, 8, 2, 8), (600, 8, 4, 13), (512, 8, 2, 45)])
def test_series_equals_rows_read_one_by_one(ianus, S, K, R, rows):
    beta = [0.5 + 0.1 * k for k in range(K)] if K > 1 else 0.7
    a, b = (ianus.Lattice(dim=2, L=8, n_samples=S, n_replicas=R, n_temps=K, seed=SEED, layout="bits64",
                          series_capacity=40) for _ in range(2))
    a.sweep("heatbath", beta, rows, 1)
    sweep, E, M, Q = a.series()
    assert len(sweep) == min(rows, 40)
    for i in range(rows):
        b.sweep("heatbath", beta, 1)
        k = i - (rows - len(sweep))
        if k < 0:
            continue
        e, m, q = b.measure(overlap=R >= 2)
        assert sweep[k] == i + 1 and np.array_equal(E[k], e) and np.array_equal(M[k], m)
        if R >= 2:
            assert np.array_equal(Q[k], q)


def test_threads_and_page_locked_arrays(ianus):
    import torch
    lats = [ianus.Lattice(dim=2, L=16, n_samples=100 + 30 * i, n_replicas=2, seed=SEED + i, layout="bits64",
                          stream=torch.cuda.Stream()) for i in range(6)]
    want = []
    for lat in lats:
        lat.sweep("heatbath", 0.9, 3)
        lat.synchronize()
        want.append(lat.measure())
    bad = []

    def read(i):
        for _ in range(50):
            got = lats[i].measure()
            if not all(np.array_equal(x, y) for x, y in zip(got, want[i])):
                bad.append(i)

    threads = [threading.Thread(target=read, args=(i,)) for i in range(6)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert not bad
    lat, pinned = lats[0], torch.empty(200, dtype=torch.int64).pin_memory()
    assert lat._lib.ianus_measure(lat._h, C.c_void_p(pinned.data_ptr()), None, None) == 0
    assert np.array_equal(pinned.numpy(), want[0][0].ravel())
