"""The one-transform-pair kernel (csrc/pd_pair.cuh): every compiled cluster shape against the FP64
oracle, the shapes a default context chooses among equal bit for bit, and resumed solves."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2006_09808_gb300 as pcs  # noqa: E402
import phantoms  # noqa: E402
from oracle import pd_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu
STEP = 1.0 / np.sqrt(4.0 / 9.0 + 8.0)
# (H, cluster size, threads, tile, member of the default family)
VARIANTS = [
    (64, 4, 128, 404, True), (64, 2, 256, 404, True), (64, 1, 512, 404, True), (64, 1, 256, 808, False),
    (128, 8, 128, 808, True), (128, 4, 256, 808, True), (128, 2, 512, 808, True), (128, 1, 512, 1616, False),
    (192, 3, 512, 1212, True), (192, 6, 256, 1212, True), (192, 12, 128, 1212, True),
    (256, 4, 512, 1616, True), (256, 8, 256, 1616, True), (256, 16, 128, 1616, True),
    (384, 8, 384, 2424, True), (512, 16, 512, 1616, True),
]
# N iterations of FP32 rounding: a few ulp (6e-8) of the result per iteration, most of it damped
N_ITER, TOL = 12, 12 * 4 * 6e-8


def problem(H, S):
    """A ragged mask that touches every border, and a field of the phantom's size."""
    pb = phantoms.volume(H, H, S, seed=H + S, lam=5e-4, n_iter=N_ITER)
    mask = (np.random.default_rng(H).random((S, H, H)) < 0.9).astype(np.uint8)
    return pb.field, mask, phantoms.magnitude_weight(mask, 3)


def solve(field, mask, lam, n_iter, weight=None, **opts):
    S, H, W = field.shape
    f, m = torch.from_numpy(field).cuda(), torch.from_numpy(mask).cuda()
    chi = torch.full_like(f, float("nan"))
    ctx = pcs.pcs_create(H, W, S, **opts)
    try:
        if weight is None:
            pcs.pcs_solve_slices(ctx, f, m, lam, STEP, STEP, n_iter, chi)
        else:
            pcs.pcs_solve_slices_weighted(ctx, f, m, torch.from_numpy(weight).cuda(), lam, STEP, STEP, n_iter, chi)
        pcs.pcs_check(ctx)
    finally:
        pcs.pcs_destroy(ctx)
    return chi.cpu().numpy()


@pytest.mark.parametrize("H,C,threads,tile,family", VARIANTS)
@pytest.mark.parametrize("tv,axis,weighted,lam", [(0, 0, False, 5e-4), (1, 1, True, 5.0)])
def test_variant_against_oracle(H, C, threads, tile, family, tv, axis, weighted, lam):
    field, mask, weight = problem(H, 2)
    opts = dict(kernel=pcs.KERNEL_STREAMING, tv=tv, b0_axis=axis)
    w = weight if weighted else None
    got = solve(field, mask, lam, N_ITER, w, cluster_size=C, threads=threads, tile=tile, **opts)
    ref = O.pd_solve(field.astype(np.float64), mask, lam, STEP, STEP, N_ITER, b0_axis=axis, tv="iso" if tv else "aniso",
                     **({"weight": weight.astype(np.float64), "tv_mask": mask} if weighted else {}))
    for s in range(2):
        assert np.linalg.norm(got[s] - ref[s]) <= TOL * np.linalg.norm(ref[s]), s
    if family:  # contexts without variant options give the same bits whatever shape they choose
        assert np.array_equal(got, solve(field, mask, lam, N_ITER, w, **opts))


@pytest.mark.parametrize("H,S", [(64, 160), (128, 80), (192, 52), (256, 40), (384, 18), (512, 10)])
def test_more_slices_than_clusters_equal_slices_alone(H, S):
    """The balanced schedule continues a split slice from its stored state: bit for bit the slice alone."""
    pb = phantoms.volume(H, H, 2, seed=9, lam=5e-4, n_iter=9)
    field = np.ascontiguousarray(np.tile(pb.field, (S // 2, 1, 1)))
    mask = np.ascontiguousarray(np.tile(pb.mask, (S // 2, 1, 1)))
    got = solve(field, mask, pb.lam, 9)
    alone = solve(pb.field, pb.mask, pb.lam, 9)
    for s in range(S):
        assert np.array_equal(got[s], alone[s % 2]), s
