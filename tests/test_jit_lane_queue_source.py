"""Every form of the lane-queue kernel (csrc/jit_sweep_lt.cuh) compiles with
the run-time compiler for sm_103a: a form that did not would silently leave
its sweeps to the slower precompiled kernels."""

import ctypes as C
import os

import pytest

from tests.test_jit_source import CSRC, _nvrtc

LUT = ",".join(str((37 * i + 11) & 127) for i in range(32))


@pytest.mark.parametrize("persist,lanes,field", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (0, 0, 2)])
@pytest.mark.parametrize("D,algo,R,L,minb", [(3, 0, 2, 64, 3), (3, 1, 1, 10, 4), (2, 1, 2, 12, 3), (2, 0, 1, 32, 4)])
def test_lane_queue_forms_compile(D, algo, R, L, minb, persist, lanes, field):
    lib = _nvrtc()
    p2 = L & (L - 1) == 0
    macros = dict(D=D, ALGO=algo, R=R, P2=int(p2), L=L, LH=(L // 2).bit_length() - 1 if p2 else 0,
                  LL=L.bit_length() - 1 if p2 else 0, MINB=minb, BLOCK=256, PERSIST=persist)
    if lanes:
        macros["LANES"] = 1
    elif field:
        macros["FIELD"] = field
        for fh in ("00", "01", "10", "11"):
            macros.update({f"LUT{fh}": LUT, f"ALWAYS{fh}": 1, f"NEED{fh}": 126})
    else:
        macros.update(LUTS=LUT, ALWAYS=0, NEED=127)
    pre = "".join(f"#define IANUS_JIT_{k} {v}\n" for k, v in macros.items()) + "#include \"jit_sweep_lt.cuh\"\n"
    hdrs = [open(os.path.join(CSRC, n), "rb").read() for n in ("common.cuh", "jit_sweep_lt.cuh")]
    prog = C.c_void_p()
    H = (C.c_char_p * 2)(*hdrs)
    N = (C.c_char_p * 2)(b"common.cuh", b"jit_sweep_lt.cuh")
    assert lib.nvrtcCreateProgram(C.byref(prog), pre.encode(), b"ianus_jit.cu", 2, H, N) == 0
    opts = (C.c_char_p * 2)(b"--gpu-architecture=sm_103a", b"-std=c++17")
    rc = lib.nvrtcCompileProgram(prog, 2, opts)
    n = C.c_size_t()
    lib.nvrtcGetProgramLogSize(prog, C.byref(n))
    log = C.create_string_buffer(n.value)
    lib.nvrtcGetProgramLog(prog, log)
    lib.nvrtcDestroyProgram(C.byref(prog))
    assert rc == 0, log.value.decode()
