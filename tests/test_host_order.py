"""The host logic of csrc/api.cu on a recording stand-in for the CUDA runtime
and the kernels (host_fake.cu): which operations are ordered before which, and
what a refused call leaves behind.  No GPU needed."""

import ctypes as C
import os
import subprocess

import pytest

import paper_0704_3573_gb300 as ianus
from paper_0704_3573_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))
ECUDA, ESTATE = 3, 6


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    b.build()
    out = tmp_path_factory.mktemp("fake")
    obj, so = str(out / "fake.o"), str(out / "fake.so")
    # without the device-side declarations of the functions that the stand-in defines
    flags = ["-O1", "-std=c++17", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "-I", b.CSRC, "-I", b.INCLUDE,
             "-D__CUDA_DEVICE_RUNTIME_API_H__"]
    subprocess.run([b.nvcc(), *b.ARCH, *flags, "-c", os.path.join(HERE, "host_fake.cu"), "-o", obj], check=True)
    objs = [os.path.join(b.BUILD_DIR, "api.o"), os.path.join(b.BUILD_DIR, "tables.o"), obj]
    # the launchers that no test here reaches
    nm = lambda how, o: {w for w in subprocess.check_output(["nm", how, o], text=True).split() if w.startswith("_ZN5ianus")}
    rest = nm("-u", objs[0]).difference(*(nm("--defined-only", o) for o in objs))
    (out / "rest.c").write_text("#include <stdlib.h>\n" + "".join(f"void {w}(void) {{ abort(); }}\n" for w in sorted(rest)))
    subprocess.run(["gcc", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-o", so, str(out / "rest.c"), *objs, "-lstdc++"],
                   check=True)
    lib = C.CDLL(so, mode=os.RTLD_LOCAL | os.RTLD_NOW)
    dp = C.POINTER(C.c_double)
    lib.fake_record.restype = C.c_char_p
    lib.fake_set.argtypes = [C.c_char_p, C.c_long]
    lib.ianus_preferred_bytes.restype = lib.ianus_required_bytes.restype = C.c_size_t
    lib.ianus_sweep.argtypes = [C.c_void_p, C.c_int32, dp, C.c_uint64, C.c_uint32]
    lib.ianus_sweep_pt.argtypes = [C.c_void_p, C.c_int32, dp, C.c_uint64, C.c_uint32, C.c_uint32]
    lib.ianus_pt_swap.argtypes = lib.ianus_destroy.argtypes = [C.c_void_p]
    lib.ianus_get_sweeps.argtypes = [C.c_void_p, C.POINTER(C.c_uint64)]
    lib.ianus_set_resident.argtypes = [C.c_void_p, C.c_int32]
    lib.ianus_measure.argtypes = [C.c_void_p] + [C.POINTER(C.c_int64)] * 3
    return lib


@pytest.fixture
def lattice(fake):
    made = []
    fake.fake_reset()

    def make(L=32, S=128, R=1, K=1, layout=1, rows=8):
        h = C.c_void_p()
        assert fake.ianus_lattice_create(C.byref(config(L, S, R, K, layout, rows)), C.byref(h)) == 0
        made.append(h)
        fake.fake_forget()
        return h

    def destroy(h):
        made.remove(h)
        fake.ianus_destroy(h)

    make.destroy = destroy
    yield make
    for h in made:
        fake.ianus_destroy(h)


def config(L=32, S=128, R=1, K=1, layout=1, rows=8):
    c = ianus.IanusConfig()
    c.abi_version, c.dim, c.L, c.n_samples, c.n_replicas, c.n_temps = ianus.ABI_VERSION, 3, L, S, R, K
    c.layout, c.occupation, c.seed, c.series_capacity = layout, 1.0, 1, rows
    return c


def betas(K):
    return (C.c_double * K)(*[1.3 - 0.1 * k for k in range(K)])


def record(lib):
    """(number, name, a, b, numbers of the operations ordered before it)"""
    ops = []
    for line in lib.fake_record().decode().splitlines():
        n, name, x, y, *before = line.split()
        ops.append((int(n), name, int(x), int(y), {int(k) for k in before}))
    return ops


@pytest.mark.parametrize("layout", [1, 2])
@pytest.mark.parametrize("measured", [0, 1])
@pytest.mark.parametrize("chains", [1, 2, 4])
def test_swaps_are_ordered_against_every_sweep(fake, lattice, layout, measured, chains):
    """A swap step writes the temperatures that the colour passes read, on every
    stream of a captured block."""
    h = lattice(K=4, layout=layout)
    fake.fake_set(b"chains", chains)
    for _ in range(3):
        assert fake.ianus_sweep_pt(h, 0, betas(4), 32, 2, 2 * measured) == 0
    ops = record(fake)
    starts = [i for i, o in enumerate(ops) if o[1] == "capture"]
    assert starts
    for i in starts:
        block = ops[i:i + [o[1] for o in ops[i:]].index("captured")]
        assert [o[1] for o in block].count("swap") >= 2
        for n, name, _, _, before in block:
            if name not in ("swap", "planes"):
                continue
            for m, other, _, _, theirs in block:
                if other in ("sweep", "sweep_bits", "measure") and m < n:
                    assert m in before, (name, n, "does not wait for", other, m)
                elif other in ("sweep", "sweep_bits") and m > n:
                    assert n in theirs, (other, m, "does not wait for", name, n)


def sweeps_done(lib, h):
    n = C.c_uint64()
    assert lib.ianus_get_sweeps(h, C.byref(n)) == 0
    return n.value


def test_a_capture_that_fails_in_words_leaves_spins_and_counters_together(fake, lattice):
    """2 sweeps, then 23 with measurements: 3 + 5 of those run before the capture of
    the rest is refused.  The bytes get the 8, and the lattice goes on."""
    h = lattice()
    fake.fake_set(b"words", 1)
    assert fake.ianus_sweep(h, 0, betas(1), 2, 0) == 0
    fake.fake_forget()
    fake.fake_set(b"fail_capture", 1)
    assert fake.ianus_sweep(h, 0, betas(1), 23, 5) == ECUDA
    names = [o[1] for o in record(fake)]
    assert names.count("sweep_bits") == 2 * 8 and sweeps_done(fake, h) == 10
    assert names[-1] == "unpack_spins"
    fake.fake_forget()
    assert fake.ianus_sweep(h, 0, betas(1), 15, 5) == 0
    names = [o[1] for o in record(fake)]
    assert "capture" in names and sweeps_done(fake, h) == 25
    assert names.index("pack_words") < names.index("capture") and names[-1] == "unpack_spins"


def test_a_launch_refused_in_words_closes_the_lattice(fake, lattice):
    h = lattice()
    fake.fake_set(b"words", 1)
    fake.fake_set(b"fail_sweep", 3)
    assert fake.ianus_sweep(h, 0, betas(1), 3, 0) == ECUDA
    assert fake.ianus_sweep(h, 0, betas(1), 3, 0) == ESTATE


@pytest.mark.parametrize("layout", [1, 2])
def test_a_resident_mode_reaches_captured_cycles(fake, lattice, layout):
    """Cycles captured under one mode are not replayed under another; setting the
    mode that is set keeps them."""
    h = lattice(layout=layout)

    def replays():
        fake.fake_forget()
        assert fake.ianus_sweep(h, 0, betas(1), 10, 5) == 0
        return [o[1] for o in record(fake)].count("graph")

    for _ in range(3):
        before = replays()
    assert before > 0
    assert fake.ianus_set_resident(h, 1) == 0 and replays() == before
    for mode in (0, 2, 3, 1):
        assert fake.ianus_set_resident(h, mode) == 0 and replays() == 0
        assert replays() + replays() > 0


def test_every_run_in_words_packs_spins_and_couplings(fake, lattice):
    """Both may have been written in the lattice's buffer since the last run."""
    h = lattice()
    fake.fake_set(b"words", 1)
    for _ in range(3):
        fake.fake_forget()
        assert fake.ianus_sweep(h, 0, betas(1), 20, 0) == 0
        names = [o[1] for o in record(fake)]
        assert "pack_words" in names[:4] and names[-1] == "unpack_spins"


@pytest.mark.parametrize("nth", [1, 2, 3])
def test_a_refused_read_waits_for_the_copies_before_it(fake, lattice, nth):
    """The page-locked block that small results pass through goes to other calls
    only when no copy writes it any more."""
    h = lattice(S=8, R=2)
    out = [(C.c_int64 * 16)() for _ in range(3)]
    fake.fake_set(b"fail_read", nth)
    assert fake.ianus_measure(h, *out) == ECUDA
    names = [o[1] for o in record(fake)]
    assert names.count("read") == nth - 1 and names[-1] == "synchronize"
    assert fake.ianus_measure(h, *out) == ESTATE


def test_the_room_beyond_the_least_is_bounded_and_given_back(fake, lattice):
    """Lattices that fill the GPU's memory still fit: those of a process take 8 GiB
    at most beyond what they need."""
    kw = dict(L=128, S=8, R=100, rows=1)  # 1.7 GB of words each
    fake.fake_set(b"words", 1)

    def room():
        c = config(**kw)
        return fake.ianus_preferred_bytes(C.byref(c)) - fake.ianus_required_bytes(C.byref(c))

    def in_words(h):
        fake.fake_forget()
        assert fake.ianus_sweep(h, 0, betas(1), 2, 0) == 0
        return "pack_words" in [o[1] for o in record(fake)]

    each = room()
    assert each > 1.6e9
    held = [lattice(**kw) for _ in range((8 << 30) // each)]
    assert all(in_words(h) for h in held)
    assert room() == 0
    late = [lattice(**kw) for _ in range(2)]
    assert not any(in_words(h) for h in late)
    lattice.destroy(late.pop(0))  # held none: gives none back
    assert room() == 0
    lattice.destroy(held.pop())
    assert room() == each and in_words(lattice(**kw)) and room() == 0
