"""The any-size transforms where their stages and kernels change: five-point stages alone, repeated and
beside others (rows and columns), direct stages whose coefficients lay 16 entries apart, and solves
small and large enough for every row kernel."""

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


@pytest.mark.parametrize("H,W", [(16, 10), (50, 40), (16, 250), (24, 500), (18, 450), (490, 16), (32, 464), (32, 272),
                                 (20, 330), (464, 20)])
def test_stages_against_oracle(H, W):
    pb = phantoms.volume(H, W, 2, seed=H + W, lam=5e-4, n_iter=N_ITER)
    got = solve(pb.field, pb.mask, pb.lam)
    for s in range(2):
        ref = O.pd_solve(pb.field[s].astype(np.float64), pb.mask[s], pb.lam, STEP, STEP, N_ITER)
        assert np.linalg.norm(got[s] - ref) <= TOL * np.linalg.norm(ref), s


@pytest.mark.parametrize("W,counts", [(258, (120, 160, 320)), (132, (120, 160)), (450, (120, 330))])
def test_row_kernels_give_the_same_bits(W, counts):
    """32 x W slices: 16 row pairs each, so these counts run two warps per pair with three and with four CTAs per
    SM, and one warp per pair, in more than one wave."""
    pb = phantoms.volume(32, W, 2, seed=W, lam=5e-4, n_iter=N_ITER)
    alone = solve(pb.field, pb.mask, pb.lam)
    for n in counts:
        got = solve(np.tile(pb.field, (n // 2, 1, 1)), np.tile(pb.mask, (n // 2, 1, 1)), pb.lam)
        for s in range(n):
            assert np.array_equal(got[s], alone[s % 2]), (n, s)
