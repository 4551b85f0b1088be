"""The history decoder's device code on the CPU (tests/emu/history_emu.cpp),
compiled with the host compiler: test infrastructure only."""
import ctypes
import os
import subprocess
import tempfile

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
PENDING = -1
_lib = None
_dir = None


def lib():
    global _lib, _dir
    if _lib is None:
        _dir = tempfile.TemporaryDirectory()
        so = os.path.join(_dir.name, "libhistory_emu.so")
        subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-shared", "-fPIC",
                        "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2506_03266_gb300", "csrc"), "-o", so,
                        os.path.join(ROOT, "tests", "emu", "history_emu.cpp")], check=True)
        _lib = ctypes.CDLL(so)
    return _lib


def decode(x, max_steps=400, m_max=255, move_thr=0, seed=0, tie=0, bal=0, sigma=False, open=False,
           all_slots=False, fill=0xFF, skew=0, order=1, threads=0):
    """Noise [shots][2][L][L] or (sigma) anyon indicators [shots][L][L]; returns
    correction, steps (PENDING where the shot is left), flag (sigma: exhausted)."""
    x = np.ascontiguousarray(x)
    n, L = x.shape[0], x.shape[-1]
    C = np.zeros((n, 2, L, L), np.uint8)
    steps = np.zeros(n, np.int32)
    flag = np.zeros(n, np.uint8)

    def p(a):
        return a.ctypes.data_as(ctypes.c_void_p)

    rc = lib().emu_history(p(x), L, n, max_steps, m_max, ctypes.c_uint64(move_thr),
                           ctypes.c_uint64(seed), tie, bal, int(sigma), int(open), int(all_slots),
                           fill, skew, ctypes.c_uint64(order), threads, p(C), p(steps), p(flag))
    if rc == -2:
        raise AssertionError("lanes of a warp or block went apart")
    assert rc == 0, rc
    return C, steps, flag
