"""Host-side decisions of the CG solves (csrc/tg_drive.h, built for the CPU tests) and, on the
GPU, the calls that they route."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from synth import initial_state, workload_params

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_05370_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "drive_check.cpp")
FIELDS = ("p", "i", "n", "g", "w", "f", "o", "l", "ux", "uy", "uz", "vx", "vy", "vz")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("drive") / "drive.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, SRC, "-o", out],
                   check=True)
    return ctypes.CDLL(out)


def _rel(a, b):
    den = np.linalg.norm(b)
    return float(np.linalg.norm(a - b) / den) if den > 0 else float(np.linalg.norm(a))


def test_small_solve_rule(lib):
    """512 voxels per SM alone or beside one other simulation; from three on, together at most
    1024."""
    def fits(n, sms, sharers):
        return bool(lib.tgd_small_fits(ctypes.c_longlong(n), sms, sharers))

    for sms in (1, 148, 152):
        most = 512 * sms
        for sharers in (1, 2):
            assert fits(most, sms, sharers) and not fits(most + 1, sms, sharers)
        for sharers in (3, 4, 8, 64):
            n = 2 * most // sharers
            assert fits(n, sms, sharers) and not fits(n + 1, sms, sharers)
    assert not fits(1, 0, 1)


@pytest.mark.parametrize("rr0", [1.0, 1e-4, 1e-8, 1e-12])
@pytest.mark.parametrize("prev,total", [(0, 50), (20, 80), (60, 62), (80, 20), (10, 120), (12, 14)])
def test_flags_are_read_few_times(lib, rr0, prev, total):
    """A residual that falls evenly, from |rhs| or from the much smaller one of a good starting
    guess.  From |rhs|: the first look, one for every 64 iterations then left (the most queued at
    once), and one more where the estimate rounds.  From any start no more than with a guess that
    doubles from two iterations to 32."""
    reads = lib.tgd_reads(total, prev, ctypes.c_double(1.0), ctypes.c_double(rr0),
                          ctypes.c_double(1e-8))
    first = prev - prev // 8 if prev else 4
    left = max(0, total - first)
    if rr0 == 1.0:
        assert reads <= 1 + -(-left // 64) + (left > 0)
    queued, guess, most = first, 2, 1
    while queued < total:
        queued, guess, most = queued + guess, min(2 * guess, 32), most + 1
    assert reads <= most


@pytest.mark.parametrize("sms", [1, 76, 148, 152])
def test_launch_shapes_follow_the_device(lib, sms):
    lib.tgd_flat_blocks.restype = ctypes.c_longlong

    def flat(want, nblocks):
        return lib.tgd_flat_blocks(ctypes.c_longlong(want), ctypes.c_longlong(nblocks), sms)

    assert flat(0, 1) == 1 and flat(1 << 30, 1 << 30) == 2 * sms
    for nblocks in (1, 5, sms, 4 * sms):
        got = flat(1 << 30, nblocks)
        assert got == min(nblocks, 2 * sms)
        assert 3 * got * 2 <= 9 * nblocks              # two sums of three components each

    def planes(zc, nblocks):
        return lib.tgd_op_planes(zc, ctypes.c_longlong(nblocks), sms)

    for zc in (1, 8):
        assert planes(zc, 4 * sms) == 2 * zc and planes(zc, 4 * sms - 1) == zc
    assert planes(9, 4 * sms) == 9


TAKEN, QUEUE, FAILED = 0, 1, 2


@pytest.mark.parametrize("error,outcome", [(0, TAKEN), (720, QUEUE), (801, QUEUE), (1, FAILED),
                                           (700, FAILED), (719, FAILED)])
def test_refused_cooperative_launch_goes_to_the_queued_kernels(lib, error, outcome):
    """A fake launch that returns a CUDA error: only the two refusals that come before anything
    ran send the solve to the queued kernels, and then the context's later solves too."""
    refused, launched = ctypes.c_int(0), ctypes.c_int(0)

    def run(fits):
        return lib.tgd_run_small(fits, ctypes.byref(refused), error, ctypes.byref(launched))

    assert run(0) == QUEUE and launched.value == 0 and not refused.value
    assert run(1) == outcome and launched.value == 1
    assert bool(refused.value) == (outcome == QUEUE)
    assert run(1) == outcome
    assert launched.value == (1 if outcome == QUEUE else 2)


@pytest.mark.gpu
@pytest.mark.parametrize("n,one_launch", [(16, True), (30, False)])
def test_concurrent_fp64_members(n, one_launch):
    """Eight FP64 members stepped by eight threads: small ones in one launch a solve as alone,
    larger ones in queued kernels (which the launch count shows), with a simulation's own
    iteration counts and its results to rounding."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count not in range(132, 211):
        pytest.skip("the sizes are chosen for 132 to 210 SMs")
    from paper_1810_05370_gb300 import Simulation
    from paper_1810_05370_gb300.batch import Batch
    shape = (n, n, n)
    P = [workload_params(rho_g=6.0 + k, rho_w=6.0 + k) for k in range(8)]
    batch = Batch([(shape, p, initial_state(shape, 40 + k)) for k, p in enumerate(P)],
                  concurrent=True, threads=8, precision="fp64")
    stats = batch.step(0.01)
    launches, its = 0, 0
    for k, p in enumerate(P):
        sim = Simulation(shape, p, initial_state(shape, 40 + k), precision="fp64")
        s = sim.step(0.01)
        launches += s["launches"]
        its += s["it_elas"]
        single, got = sim.numpy(), batch.numpy(k)
        sim.close()
        for f in FIELDS:
            if one_launch:
                assert np.array_equal(got[f], single[f]), (k, f)
            else:
                # two orders of the same sums: rounding, times the condition of the solve for u
                # and, in v = (u' - u) / dt, the difference's own
                gate = 1e-10
                if f[0] == "v":
                    gate *= 2 * np.linalg.norm(single["u" + f[1]]) / (0.01 * np.linalg.norm(single[f]))
                assert _rel(got[f], single[f]) <= gate, (k, f)
    assert stats["it_elas_total"] == its
    assert (stats["launches"] == launches) if one_launch else (stats["launches"] > 3 * launches)
    batch.close()
