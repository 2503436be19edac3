"""FP64 spectral preconditioner in any units: elasticity scaled by a power of two.

CPU: the scale that the z pass takes (csrc/tg_fpconv.cuh).  GPU: E, eta and the force multiplied
by one power of two leave the displacement as it is, bit for bit."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from synth import initial_state, workload_params

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_05370_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "scale_check.cpp")


def test_scale(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path / "scale.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, SRC, "-o", out],
                   check=True)
    lib = ctypes.CDLL(out)
    e = np.arange(-1022, 1024)
    x = np.concatenate([np.ldexp(1.0, e), np.ldexp(1.75, e), [0.0, 2.0 ** -1030]])
    got = np.empty_like(x)
    p = ctypes.POINTER(ctypes.c_double)
    lib.tgs_pow2_scale(x.ctypes.data_as(p), got.ctypes.data_as(p), ctypes.c_long(x.size))
    want = np.ldexp(1.0, np.clip(-e, -880, 880))
    assert np.array_equal(got, np.concatenate([want, want, [1.0, 1.0]]))
    scaled = x[:-2] * got[:-2]           # six factors up to 2^20 apart
    assert np.all(np.ldexp(scaled, 20) ** 6 < np.inf)
    assert np.all(np.ldexp(scaled, -20) ** 6 >= 2.0 ** -1022)


@pytest.mark.gpu
@pytest.mark.parametrize("precond", [1, 2])
@pytest.mark.parametrize("k", [-220, -190, 190, 220])
def test_displacement_does_not_depend_on_the_units(precond, k):
    """2^k times E, eta and zeta.  The squares in the solves' scalars stay in range at these k; the
    products of six diagonals of about 2^27 each do not unless they are scaled."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1810_05370_gb300 import Simulation
    n, u, its = (16, 8, 32), [], []
    for f in (1.0, 2.0 ** k):
        P = workload_params(precond_elas=precond)
        P = dict(P, E_scale=P["E_scale"] * f, eta=[v * f for v in P["eta"]], zeta=P["zeta"] * f)
        sim = Simulation(n, P, initial_state(n, 6), precision="fp64")
        u.append([sim.state[q].cpu().numpy() for q in ("ux", "uy", "uz")])
        its.append(sim.init_stats["it_elas"])
        sim.close()
    assert its[0] == its[1]
    for a, b in zip(*u):
        assert np.linalg.norm(a) > 0 and np.array_equal(a, b)
