"""A batch handle whose calls have other slice counts than its first: each count runs in the shape that
suits it, with the bits of the first."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2006_09808_gb300 as pcs  # noqa: E402
import phantoms  # noqa: E402

pytestmark = pytest.mark.gpu
N_ITER = 20


@pytest.mark.parametrize("autotune", [True, False])
def test_shape_follows_each_call(autotune):
    pb = phantoms.volume(256, 256, 64, seed=3, lam=5e-4, n_iter=N_ITER)
    f, m = torch.from_numpy(pb.field.copy()).cuda(), torch.from_numpy(pb.mask.copy()).cuda()

    def solve(batch, S):
        chi = torch.full((S, 256, 256), float("nan"), device="cuda")
        pcs.pcs_batch_solve(batch, [(f[:S], m[:S], pb.lam, chi)], N_ITER)
        pcs.pcs_batch_check(batch)
        return chi.cpu().numpy(), pcs.pcs_batch_tuning(batch, 256, 256)["cluster_size"]

    for first, then in ((1, 64), (64, 1)):
        batch = pcs.pcs_batch_create(autotune=autotune)
        try:
            a, shape_a = solve(batch, first)
            b, shape_b = solve(batch, then)
            c, shape_c = solve(batch, first)
        finally:
            pcs.pcs_batch_destroy(batch)
        # 64 slices need the SM time of the 4-CTA shape, a slice alone the speed of a larger one
        by_count = {first: shape_a, then: shape_b}
        assert by_count[64] == 4 and by_count[1] > 4 and shape_c == shape_a
        assert np.array_equal(a, c)
        k = min(first, then)
        assert np.isfinite(b).all() and np.array_equal(a[:k], b[:k])
