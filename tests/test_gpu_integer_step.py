"""The RK4 step on the integer pipes (csrc/lorenz_int.cuh) on the GPU, bit-exact against the oracle where it can
go wrong: gammas and step sizes at and beyond the range it takes, states at and beyond its grids' limits, states
with few significand bits (ties), zeros and negatives, and long chains.  Every value it cannot take is done in
binary64, so each comparison is for equality of every byte."""
import numpy as np
import pytest
import torch

import oracle
import synth_inputs as si
from gpu_util import host, host_u16, to_dev

pytestmark = pytest.mark.gpu

fhd = pytest.importorskip("paper_2505_07158_gb300")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _attractor(g, gamma, count, h=0.01):
    s = oracle.rk4_trajectory([g.uniform(1, 20), g.uniform(1, 20), g.uniform(5, 40), g.uniform(1, 20)], gamma, 400, h)
    return s[-1 - np.arange(count) * 3]


def _pairs(IR, gamma, n, h=0.01, shape=(24, 40, 3)):
    """The n worker pairs from IR (one pair per warp on the integer pipes) against the oracle's Algorithm 2."""
    D_ref, B_ref = oracle.keystream(IR, gamma, *shape, n, h)
    D, B = fhd.fhd_keystream(to_dev(np.ascontiguousarray(IR)), gamma, *shape, n_workers=n, rk4_h=h)
    assert np.array_equal(host_u16(D), D_ref)
    assert np.array_equal(host(B), B_ref)


@pytest.mark.parametrize("gamma", [-1.52, -0.9123, -0.06, 0.7, 1.999, 2.0, -2.5, -1.0, -0.5, 0.0, -3e-3, -1e-3, 1e-300])
def test_gammas_in_and_out_of_range(gamma):
    g = si.rng(11)
    _pairs(_attractor(g, -0.9, 8), gamma, 4)


@pytest.mark.parametrize("h", [1e-4, 7.9e-4, 8.1e-4, 1e-3, 0.005, 0.0078125, 0.01, 0.02, 0.0399, 0.041, 0.05])
def test_step_sizes_in_and_out_of_range(h):
    g = si.rng(12)
    _pairs(_attractor(g, -0.9, 8), -0.7315, 4, h)


def test_states_at_the_limits():
    """Each variable at, just inside and just outside its range and its smallest magnitude, exact powers of two,
    small integers (few significand bits), zeros, negative zeros and negatives, one per chain."""
    g = si.rng(13)
    base = _attractor(g, -0.9, 1)[0]
    rows = []
    for v, lim in enumerate((32.0, 32.0, 64.0, 256.0)):
        for x in (np.nextafter(lim, 0), lim, np.nextafter(lim, 1e9), 2.0 ** -9, np.nextafter(2.0 ** -9, 0), 2.0 ** -7,
                  2.0 ** -12, 1e-30, 1.0, 3.0, 8.0, 0.0, -0.0, 5e-324, 1000.0):
            for sign in (1.0, -1.0):
                s = base.copy()
                s[v] = sign * x
                rows.append(s)
    rows += [np.zeros(4), np.array([1.0, 1.0, 1.0, 1.0]), np.array([2.0, -3.0, 17.0, 9.0]),
             np.array([1e3, -1e3, 1e3, 1e3])]
    _pairs(np.array(rows), -0.9123, len(rows) // 2, shape=(64, 80, 3))


@pytest.mark.parametrize("seed", range(6))
def test_long_master_chains(seed):
    """1024 workers: 2048 chained steps of LHCS_m from a reconstructed state, IR and the last state."""
    g = si.rng(100 + seed)
    gamma = float(g.uniform(-1.52, -0.06))
    v = [float(g.uniform(-50, 50)) for _ in range(4)]
    H = g.integers(0, 256, size=32, dtype=np.uint8).tobytes()
    IR_ref, last = oracle.master(v, H, gamma, n=1024)
    st = to_dev(np.array(v + [gamma], np.float64))
    IR = fhd.fhd_master(st, to_dev(np.frombuffer(H, np.uint8).copy()), n_workers=1024)
    assert np.array_equal(host(IR).view(np.uint64), np.asarray(IR_ref).view(np.uint64))
    assert np.array_equal(host(st)[:4].view(np.uint64), np.asarray(last).view(np.uint64))


@pytest.mark.parametrize("n", [303, 304, 305, 608, 609])
def test_worker_pairs_around_the_one_pair_launch_limit(n):
    """Pair counts on both sides of the limit (608) between the integer one-pair kernel and the binary64 one."""
    g = si.rng(n)
    IR = np.column_stack([g.uniform(0, 20, 2 * n), g.uniform(0, 20, 2 * n), g.uniform(0, 40, 2 * n), g.uniform(0, 20, 2 * n)])
    _pairs(IR, -0.8, n, shape=(90, 110, 3))


@pytest.mark.parametrize("count", [1, 7, 33])
def test_trajectories_of_a_batch_with_other_gammas(count):
    """Frames of streams with their own gammas in one call, some out of the integer step's range."""
    g = si.rng(count)
    n = 8
    c = fhd.Cipher(bytes(32), n_workers=n)
    items, refs, frames = [], [], []
    for k in range(count):
        ic = np.array([g.uniform(0, 20), g.uniform(0, 20), g.uniform(0, 40), g.uniform(0, 20),
                       (-1.0, 0.0, -0.9)[k % 3] if k % 2 else g.uniform(-1.5, -0.1)], np.float64)
        F = si.uniform_frame(20 + k % 5, 30 + 3 * (k % 4), 3, seed=k)
        sid = c.open_stream()
        c.import_state(sid, ic.tobytes() + bytes(8))
        src = to_dev(F)
        items.append((sid, src, torch.empty_like(src), torch.empty(32, dtype=torch.uint8, device=src.device)))
        refs.append(oracle.Stream(ic, n=n))
        frames.append(F)
    c.encrypt_frames(items)
    for (_, _, E, H), ref, F in zip(items, refs, frames):
        E_ref, H_ref = ref.encrypt(F)
        assert np.array_equal(host(E), E_ref) and bytes(host(H)) == H_ref
    c.close()


def test_states_at_the_edges_of_each_grid():
    """Each variable round its range and round the smallest magnitudes of the grids, in both chains of a pair."""
    g = si.rng(17)
    base = _attractor(g, -0.9, 1)[0]
    rows = []
    for v, lim in enumerate((28.0, 30.0, 50.0, 216.0)):
        for x in (lim, 2.0 ** -9, 2.0 ** -10, 2.0 ** -11, 2.0 ** -12, 2.0 ** -13, 1.0 + 2.0 ** -20, 1.0 + 2.0 ** -33):
            for y in (np.nextafter(x, 0), x, np.nextafter(x, 1e9)):
                for sign in (1.0, -1.0):
                    s = base.copy()
                    s[v] = sign * y
                    rows.append(s)
    _pairs(np.array(rows), -0.9123, len(rows) // 2, shape=(64, 80, 3))
