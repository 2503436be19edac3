"""The cooperative solves' time-bounded waits.

CPU: the wait and the publication of the result (csrc/tg_wait.cuh, built for the host) over
orders in which a block gives up and the others finish.  GPU: a limit that every wait exceeds."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from synth import initial_state, workload_params

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_05370_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "wait_check.cpp")
ARRIVE, WAIT, LEAVE = 0, 1, 2
RUNNING, CONVERGED, TIMEOUT = 0, 1, 5


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("waits") / "waits.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, SRC, "-o", out],
                   check=True)
    return ctypes.CDLL(out)


class Launch:
    def __init__(self, lib, blocks, words=(0, 0)):
        self.lib, self.blocks = lib, blocks
        self.words = (ctypes.c_uint * 2)(*words)
        self.status = ctypes.c_int(RUNNING)

    def __call__(self, what, rnd=0, limit_ns=10**9):
        return bool(self.lib.tgw_step(self.words, ctypes.byref(self.status), what,
                                      ctypes.c_uint(rnd), ctypes.c_uint(self.blocks),
                                      ctypes.c_ulonglong(limit_ns)))


@pytest.mark.parametrize("blocks", [1, 2, 7])
def test_last_block_publishes_once(lib, blocks):
    L = Launch(lib, blocks)
    for launch in range(2):               # the second starts from the words the first left
        L.status.value = RUNNING
        for rnd in (1, 2, 3):
            for _ in range(blocks):
                L(ARRIVE)
            assert all(L(WAIT, rnd) for _ in range(blocks))
        assert [L(LEAVE) for _ in range(blocks)] == [False] * (blocks - 1) + [True]
        assert L.status.value == CONVERGED and tuple(L.words) == (0, 0)


@pytest.mark.parametrize("gives_up", [0, 1, 2])
def test_late_block_does_not_hide_a_timeout(lib, gives_up):
    """The last wait of a solve: one block gives up before the latest arrives, the rest pass and
    finish.  The solve stays timed out, whichever block it was."""
    L = Launch(lib, 3)
    L(ARRIVE), L(ARRIVE)                  # the block that gives up is one of these
    assert not L(WAIT, 1, limit_ns=1000)
    L(ARRIVE)                             # just too late for it
    for b in range(3):
        if b != gives_up:
            assert L(WAIT, 1) and not L(LEAVE)
    assert L.status.value == TIMEOUT


def test_rounds_wrap(lib):
    L = Launch(lib, 2, words=(2**32 - 2, 0))
    L(ARRIVE)
    assert not L(WAIT, 2**31, limit_ns=0)
    L(ARRIVE)
    assert L(WAIT, 2**31)                 # 2 * 2^31 = 0 modulo 2^32


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(16, 16, 16), (36, 20, 12)])
def test_wait_limit_reports_timeout(oracle, n):
    """FP64 members whose solves are one cooperative launch each: with a limit that every wait
    exceeds the step returns TG_ERR_TIMEOUT and the batch refuses further steps; other contexts
    go on."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1810_05370_gb300 import _tg
    from paper_1810_05370_gb300.batch import Batch
    P = workload_params()

    def make():
        return Batch([(n, P, initial_state(n, 31))], concurrent=True, precision="fp64")

    batch = make()
    batch.set_timeout(1)                  # 1 ns
    with pytest.raises(_tg.TGError) as e:
        batch.step(0.01)
    assert e.value.status == _tg.TG_ERR_TIMEOUT
    with pytest.raises(_tg.TGError) as e:
        batch.step(0.01)
    assert e.value.status == _tg.TG_ERR_STATE
    batch.close()
    batch = make()
    batch.step(0.01)
    got = batch.numpy(0)
    ref = initial_state(n, 31)
    oracle.init(n, P, ref)
    oracle.step(n, P, 0.01, ref)
    for k in ("p", "i", "n", "g", "w", "f", "o", "l", "ux", "uy", "uz", "vx", "vy", "vz"):
        den = np.linalg.norm(ref[k])
        assert np.linalg.norm(got[k] - ref[k]) <= 1e-10 * (den if den > 0 else 1.0), k
    batch.close()
