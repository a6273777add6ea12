"""The any-size row kernel where its lane groups and stages change: short rows that fill the GPU with
one warp per row pair (a slice alone takes two), the largest prime stages, a prime after a prime, and
the six-point stage beside 4s and 3s."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2006_09808_gb300 as pcs  # noqa: E402
import phantoms  # noqa: E402
from oracle import pd_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu
STEP = 1.0 / np.sqrt(4.0 / 9.0 + 8.0)
# FP32 rounding of N iterations: a few ulp (6e-8) per iteration; a direct prime stage sums up to 30 terms
N_ITER, TOL = 8, 8 * 8 * 6e-8


def solve(field, mask, lam):
    f, m = torch.from_numpy(np.ascontiguousarray(field)).cuda(), torch.from_numpy(np.ascontiguousarray(mask)).cuda()
    chi = torch.full_like(f, float("nan"))
    pcs.pcs_solve_slices_generic(f, m, lam, STEP, STEP, N_ITER, chi)
    return chi.cpu().numpy()


def check(got, pb, s):
    ref = O.pd_solve(pb.field[s].astype(np.float64), pb.mask[s], pb.lam, STEP, STEP, N_ITER)
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref), s


@pytest.mark.parametrize("H,W", [(64, 122), (24, 118), (16, 10), (32, 70), (48, 486), (18, 54), (20, 494), (12, 286)])
def test_stage_plans_against_oracle(H, W):
    assert pcs.pcs_supported_generic(H, W)
    pb = phantoms.volume(H, W, 2, seed=H + W, lam=5e-4, n_iter=N_ITER)
    got = solve(pb.field, pb.mask, pb.lam)
    for s in range(2):
        check(got[s], pb, s)


def test_one_warp_per_pair_equals_two():
    """44 slices of 128 x 132 are 2816 row pairs (one warp each); a slice alone is 64 (two warps each)."""
    pb = phantoms.volume(128, 132, 2, seed=5, lam=5e-4, n_iter=N_ITER)
    got = solve(np.tile(pb.field, (22, 1, 1)), np.tile(pb.mask, (22, 1, 1)), pb.lam)
    for s in range(2):
        check(got[s], pb, s)
        alone = solve(pb.field[s:s + 1], pb.mask[s:s + 1], pb.lam)
        for k in range(s, 44, 2):
            assert np.array_equal(got[k], alone[0]), k
