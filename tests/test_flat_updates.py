"""The queued FP64 solves' flat two-voxel updates and the size from which they run.

Solves of up to 512 voxels per SM are one launch each, so an odd voxel count reaches the updates'
last single voxel only above that size, which depends on the device."""
import numpy as np
import pytest

from synth import initial_state, workload_params

pytestmark = pytest.mark.gpu
FIELDS = ("p", "i", "n", "g", "w", "f", "o", "l", "ux", "uy", "uz", "vx", "vy", "vz")
TOL, DT = 1e-10, 0.01


@pytest.fixture(scope="module")
def limit():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return 512 * torch.cuda.get_device_properties(0).multi_processor_count


def centred_on_the_last_voxel(n):
    """The workload's state, the periodic box shifted so that the tumor's densest voxel is the last
    in memory: every field changes there."""
    st = initial_state(n, 4)
    at = np.unravel_index(np.argmax(st["i"]), st["i"].shape)
    shift = [s - 1 - a for s, a in zip(st["i"].shape, at)]
    return {k: np.ascontiguousarray(np.roll(v, shift, (0, 1, 2))) for k, v in st.items()}


def against_the_oracle(oracle, n, P):
    """Two steps; returns the launches of the second."""
    from paper_1810_05370_gb300 import Simulation
    ref = centred_on_the_last_voxel(n)
    s0 = oracle.init(n, P, ref)
    want = [oracle.step(n, P, DT, ref) for _ in range(2)]
    sim = Simulation(n, P, centred_on_the_last_voxel(n), precision="fp64")
    got = [sim.step(DT) for _ in range(2)]
    out = sim.numpy()
    assert sim.init_stats["it_elas"] == s0["it_elas"]
    for a, b in zip(got, want):
        assert a["it_elas"] == b["it_elas"] and a["it_diff"] == b["it_diff"]
    for k in FIELDS:
        den = np.linalg.norm(ref[k])
        assert np.linalg.norm(out[k] - ref[k]) <= TOL * (den if den > 0 else 1.0), k
    sim.close()
    return got[1]["launches"]


def test_odd_count_above_the_one_launch_size(oracle, limit):
    nz = limit // (47 * 41) + 1
    nz += 1 - nz % 2
    n = (47, 41, nz)
    assert n[0] * n[1] * n[2] % 2 == 1 and n[0] * n[1] * n[2] > limit
    against_the_oracle(oracle, n, workload_params())


def test_one_launch_size_is_the_devices(oracle, limit):
    """512 voxels on each SM: the largest solve of one launch; one plane more: queued kernels."""
    P, sms = workload_params(), limit // 512
    below = against_the_oracle(oracle, (64, 8, sms), P)
    above = against_the_oracle(oracle, (64, 8, sms + 1), P)
    assert below < 40 < above
