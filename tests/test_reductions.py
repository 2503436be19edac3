"""The CG solves' reductions, flat vector updates and scalar decisions.

CPU: the power-of-two scale of a refinement's inner right-hand side and the convergence test
from the squares of the norms (csrc/tg_fpconv.cuh, built for the host) against their
definitions.  GPU: solves and steps on grids whose voxel count leaves remainders everywhere --
odd counts (the two-voxel accesses' tail), counts that are not multiples of four, fewer voxels
than one block has threads -- against the CPU oracle, with its iteration counts."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from synth import initial_state, workload_params

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1810_05370_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "cg_scalar_check.cpp")
FIELDS = ("p", "i", "n", "g", "w", "f", "o", "l", "ux", "uy", "uz", "vx", "vy", "vz")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    out = str(tmp_path_factory.mktemp("cgs") / "cgs.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared",
                    "-I", CSRC, SRC, "-o", out], check=True)
    return ctypes.CDLL(out)


def _p(a, t=ctypes.c_double):
    return a.ctypes.data_as(ctypes.POINTER(t))


def test_scale_is_the_nearest_power_of_two(lib):
    rng = np.random.default_rng(0)
    powers = np.ldexp(1.0, np.arange(-1022, 1024))
    x = np.concatenate([np.exp(rng.uniform(-700, 700, 20000)), powers,
                        np.nextafter(powers, 0.0), np.nextafter(powers, np.inf)])
    got = np.empty_like(x)
    lib.tgr_pow2_inv_root(_p(x), _p(got), ctypes.c_long(x.size))
    # rint(log2(x) / 2) from the exact exponent and significand x = m 2^e, 1 <= m < 2: the
    # halves' distance decides, and only m = 1 with e odd is a tie (to even)
    m, e = np.frexp(x)
    m, e = 2 * m, e - 1
    k = np.where(e % 2 == 0, e // 2, (e + 1) // 2)
    tie = (e % 2 == 1) & (m == 1.0) & (k % 2 == 1)
    assert np.array_equal(got, np.ldexp(1.0, -(k - tie)))
    typical = (x > 1e-200) & (x < 1e200) & (np.abs(np.log2(m) - 0.5) < 0.49)
    assert np.array_equal(got[typical], np.exp2(-np.rint(0.5 * np.log2(x[typical]))))


def test_power_of_two_reciprocal(lib):
    x = np.ldexp(1.0, np.arange(-1022, 1023))
    got = np.empty_like(x)
    lib.tgr_pow2_recip(_p(x), _p(got), ctypes.c_long(x.size))
    assert np.array_equal(got, 1.0 / x)


def test_convergence_test_from_the_squares(lib):
    rng = np.random.default_rng(1)
    n = 60000
    rtol = 10.0 ** rng.uniform(-14, -1, n)
    bb = 10.0 ** rng.uniform(-250, 250, n)
    rr = rtol * rtol * bb * (1.0 + rng.choice([-1, 1], n) * 10.0 ** rng.uniform(-17, 0.5, n))
    special = [(0.0, 1e-8, 1.0), (1.0, 0.0, 1.0), (0.0, 0.0, 1.0), (1e-320, 1e-8, 1e-300),
               (1.0, 1e-8, 1e300), (1e300, 1.0, 1e300), (4.0, 1.0, 4.0)]
    rr, rtol, bb = (np.concatenate([a, [s[q] for s in special]])
                    for q, a in ((0, rr), (1, rtol), (2, bb)))
    rr = np.abs(rr)
    got = np.empty(rr.size, np.int32)
    lib.tgr_norm_met(_p(rr), _p(rtol), _p(bb), _p(got, ctypes.c_int), ctypes.c_long(rr.size))
    assert np.array_equal(got == 1, np.sqrt(rr) <= rtol * np.sqrt(bb))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(5, 5, 5), (9, 7, 5), (33, 9, 7), (35, 17, 13)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_remainders_against_the_oracle(oracle, n, precision):
    against_the_oracle(oracle, n, precision)


@pytest.mark.gpu
def test_operator_blocks_of_two_chunks(oracle):
    """666 blocks of one plane: the FP32 operator takes two planes a block, the last block one."""
    against_the_oracle(oracle, (64, 72, 37), "mixed")


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(16, 8, 4), (32, 16, 8), (8, 32, 32), (64, 16, 64)])
def test_narrow_z_tiles(oracle, n):
    """The FP32 z pass of short columns in narrow tiles: half spectra of 5, 9, 17 and 33 modes (a
    partial tile, a last tile of one), columns of 4 to 64."""
    against_the_oracle(oracle, n, "mixed", workload_params(precond_elas=2))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(32, 32, 8), (64, 128, 4), (128, 64, 32), (256, 32, 4)])
def test_compile_time_lines(oracle, n):
    """The FP32 x and y passes' compile-time line lengths, 32 to 256 and 32 to 128, each beside
    another length on the other axis."""
    against_the_oracle(oracle, n, "mixed", workload_params(precond_elas=2))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(4, 8, 16), (16, 4, 128), (32, 128, 8), (64, 16, 64),
                               (256, 32, 4)])
def test_fp64_transform_lengths(oracle, n):
    """The FP64 transforms' folded twiddles and the z pass's one quotient per mode: first stages
    of radix 2, 4, 8 and 16, a radix-16 stage after each, on every axis."""
    against_the_oracle(oracle, n, "fp64", workload_params(precond_elas=2))


@pytest.mark.gpu
@pytest.mark.parametrize("n", [(64, 64, 19), (64, 64, 20), (47, 33, 50)])
def test_cooperative_solve_size_limit(oracle, n):
    """512 voxels on each of 152 SMs: the largest FP64 Jacobi solve of one launch, the smallest
    above it, and a last block of part of its threads."""
    against_the_oracle(oracle, n, "fp64")


def against_the_oracle(oracle, n, precision, P=None):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1810_05370_gb300 import Simulation
    P, dt, tol = P or workload_params(), 0.01, 1e-10 if precision == "fp64" else 1e-5
    ref = initial_state(n, 4)
    s0 = oracle.init(n, P, ref)
    st = [oracle.step(n, P, dt, ref) for _ in range(2)]
    sim = Simulation(n, P, initial_state(n, 4), precision=precision)
    got = [sim.step(dt) for _ in range(2)]
    out = sim.numpy()
    if precision == "fp64":
        assert sim.init_stats["it_elas"] == s0["it_elas"]
        for a, b in zip(got, st):
            assert a["it_elas"] == b["it_elas"] and a["it_diff"] == b["it_diff"]
    for k in FIELDS:
        den = np.linalg.norm(ref[k])
        gate = tol
        if precision == "mixed" and k[0] == "v":
            # v = (u' - u) / dt: the difference two displacements within tol leave in it
            gate = 2 * tol * np.linalg.norm(ref["u" + k[1]]) / (dt * den)
        err = np.linalg.norm(out[k] - ref[k]) / (den if den > 0 else 1.0)
        assert err <= gate, (k, err)
    sim.close()
