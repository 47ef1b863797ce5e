"""Long chains of the RK4 step (LHCS_m and worker pairs of 1,024 workers) that leave the integer step's ranges for a while
or for good, against the oracle: every byte of the iterates, the last state and the keystream is equal (of a chain that
overflows, up to there; a NaN is a NaN)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2505_07158_gb300 as fhd

pytestmark = pytest.mark.gpu


def same(got, ref):
    got, ref = np.ascontiguousarray(got), np.ascontiguousarray(ref)
    nan = np.isnan(ref)
    return np.array_equal(np.isnan(got), nan) and np.array_equal(got.view(np.uint64)[~nan], ref.view(np.uint64)[~nan])


def check_master(v, gamma, n, h=0.01, seed=1):
    g = np.random.default_rng(seed)
    H = g.integers(0, 256, size=32, dtype=np.uint8).tobytes()
    ref, last = oracle.master(list(v), H, gamma, n=n, h=h)
    st = torch.tensor([*v, gamma], dtype=torch.float64, device="cuda")
    IR = fhd.fhd_master(st, torch.from_numpy(np.frombuffer(H, np.uint8).copy()).cuda(), n_workers=n, rk4_h=h)
    assert same(IR.cpu().numpy(), ref) and same(st.cpu().numpy()[:4], last)


@pytest.mark.parametrize("gamma", [-0.02, 0.1, 0.2, 0.3, 0.5, 0.9, 1.9])
@pytest.mark.parametrize("seed", range(2))
def test_master_chains_that_leave_the_ranges(gamma, seed):
    g = np.random.default_rng(seed)
    check_master(g.uniform(-50, 50, 4), gamma, 1024, seed=seed)


@pytest.mark.parametrize("gamma,scale", [(-0.9123, 10.0), (-0.9123, 3.0), (-0.9123, 0.0), (0.2, 1.0)])
def test_worker_pairs_that_leave_the_ranges(gamma, scale):
    """Far states that come back to the attractor, states at the origin, which never leave it, and a gamma beyond its."""
    g = np.random.default_rng(int(scale))
    IR = g.uniform(0, 1, (8, 4)) * [20, 20, 40, 20] * scale
    D_ref, B_ref = oracle.keystream(IR, gamma, 60, 100, 3, 4, 0.01)
    D, B = fhd.fhd_keystream(torch.from_numpy(IR).cuda(), gamma, 60, 100, 3, n_workers=4)
    assert np.array_equal(D.cpu().numpy().view(np.uint16), D_ref) and np.array_equal(B.cpu().numpy().reshape(-1), np.asarray(B_ref).reshape(-1))


@pytest.mark.parametrize("gamma,h", [(-0.9123, 8.1e-4), (-0.0041, 8.1e-4), (0.2499, 8.1e-4), (-1.9999, 8.1e-4), (-0.9123, 0.02),
                                     (-1.52, 0.0399), (-0.9123, 0.0399), (-0.0601, 0.0399), (-1.9999, 0.0399), (-0.0041, 0.01),
                                     (0.0041, 0.01), (-1.9999, 0.01), (-0.06, 0.01)])
@pytest.mark.parametrize("seed", range(2))
def test_master_chains_at_the_ends_of_the_integer_steps_range(gamma, h, seed):
    """Step sizes and gammas just inside the range that the integer step takes: its shadows' error bounds scale with both,
    and a bound that is too small shows in a rare step only."""
    g = np.random.default_rng(100 + seed)
    check_master(g.uniform(-50, 50, 4), gamma, 1024, h, seed)
