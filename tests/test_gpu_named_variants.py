"""The variants that only options reach, named in full (cluster size, kernel, threads, tile) and checked to
be what ran: the resident kernels with more slices than clusters, and the half-spectrum kernels' isotropic,
weighted, resumed and balanced forms; and the default kernel's resume and regularisation range."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2006_09808_gb300 as pcs  # noqa: E402
import phantoms  # noqa: E402
from oracle import pd_oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu
STEP = 1.0 / np.sqrt(4.0 / 9.0 + 8.0)
# N iterations of FP32 rounding: a few ulp (6e-8) of the result per iteration, most of it damped
N_ITER, TOL = 12, 12 * 4 * 6e-8
# (H, cluster size, threads, tile, slices that outnumber the resident clusters)
RESIDENT = [(64, 1, 256, 808, 620), (128, 4, 256, 816, 80), (256, 8, 256, 1616, 20), (256, 8, 512, 808, 20)]
HALF_SPECTRUM = [(128, 1, 256, 816, 310), (128, 2, 256, 816, 160), (192, 2, 256, 1212, 160), (256, 2, 256, 1616, 80),
                 (256, 4, 256, 1616, 80), (256, 4, 512, 816, 40), (256, 4, 512, 1608, 40), (384, 4, 256, 1224, 40),
                 (384, 4, 384, 1224, 40), (512, 8, 256, 1616, 20), (512, 8, 512, 1616, 20)]


def problem(H, S):
    """A ragged mask that touches every border, and a field of the phantom's size."""
    pb = phantoms.volume(H, H, 2, seed=H, lam=5e-4, n_iter=N_ITER)
    mask = (np.random.default_rng(H).random((2, H, H)) < 0.9).astype(np.uint8)
    reps = ((S + 1) // 2, 1, 1)
    weight = phantoms.magnitude_weight(mask, 3).astype(np.float32)
    return [np.ascontiguousarray(np.tile(a, reps)[:S]) for a in (pb.field, mask, weight)]


def solve(field, mask, lam=5e-4, weight=None, n_iter=N_ITER, every=0, **opts):
    S, H, W = field.shape
    f, m = torch.from_numpy(field).cuda(), torch.from_numpy(mask).cuda()
    chi = torch.full_like(f, float("nan"))
    ctx = pcs.pcs_create(H, W, S, **opts)
    try:
        if every:
            pcs.pcs_solve_slices_monitored(ctx, f, m, lam, STEP, STEP, n_iter, every, 0.0, chi)
        elif weight is None:
            pcs.pcs_solve_slices(ctx, f, m, lam, STEP, STEP, n_iter, chi)
        else:
            pcs.pcs_solve_slices_weighted(ctx, f, m, torch.from_numpy(weight).cuda(), lam, STEP, STEP, n_iter, chi)
        pcs.pcs_check(ctx)
        ran = pcs.pcs_last_variant(ctx)
        for k in ("cluster_size", "threads", "tile"):
            assert not opts.get(k) or ran[k] == opts[k], (ran, opts)
    finally:
        pcs.pcs_destroy(ctx)
    return chi.cpu().numpy()


def check(got, field, mask, lam=5e-4, weight=None, tv=0, axis=0):
    ref = O.pd_solve(field.astype(np.float64), mask, lam, STEP, STEP, N_ITER, b0_axis=axis, tv="iso" if tv else "aniso",
                     **({} if weight is None else {"weight": weight.astype(np.float64), "tv_mask": mask}))
    for s in range(len(field)):
        assert np.linalg.norm(got[s] - ref[s]) <= TOL * np.linalg.norm(ref[s]), s


@pytest.mark.parametrize("H,C,threads,tile,S", RESIDENT)
@pytest.mark.parametrize("tv,axis", [(0, 0), (1, 1)])
def test_resident_variant(H, C, threads, tile, S, tv, axis):
    opts = dict(kernel=pcs.KERNEL_RESIDENT, cluster_size=C, threads=threads, tile=tile, tv=tv, b0_axis=axis)
    field, mask, _ = problem(H, S)
    got = solve(field, mask, **opts)
    check(got[:2], field[:2], mask[:2], tv=tv, axis=axis)
    alone = solve(field[:2], mask[:2], **opts)
    for s in range(S):  # every cluster solves several slices in turn, each from a zero start
        assert np.array_equal(got[s], alone[s % 2]), s


@pytest.mark.parametrize("H,C,threads,tile,S", HALF_SPECTRUM)
@pytest.mark.parametrize("tv,axis,weighted", [(0, 0, False), (1, 1, True), (1, 0, False)])
def test_half_spectrum_variant(H, C, threads, tile, S, tv, axis, weighted):
    opts = dict(kernel=pcs.KERNEL_STREAMING, cluster_size=C, threads=threads, tile=tile, tv=tv, b0_axis=axis)
    field, mask, weight = problem(H, 2)
    w = weight if weighted else None
    got = solve(field, mask, weight=w, **opts)
    check(got, field, mask, weight=w, tv=tv, axis=axis)
    if not weighted:
        assert np.array_equal(got, solve(field, mask, every=5, **opts))  # resumed from its stored state


@pytest.mark.parametrize("H,C,threads,tile,S", HALF_SPECTRUM)
def test_half_spectrum_variant_balanced(H, C, threads, tile, S):
    """More slices than clusters, weighted and isotropic: the balanced schedule's hand-over keeps every bit."""
    opts = dict(kernel=pcs.KERNEL_STREAMING, cluster_size=C, threads=threads, tile=tile, tv=1)
    field, mask, weight = problem(H, S)
    got = solve(field, mask, weight=weight, **opts)
    alone = solve(field[:2], mask[:2], weight=weight[:2], **opts)
    for s in range(S):
        assert np.array_equal(got[s], alone[s % 2]), s


@pytest.mark.parametrize("H,S", [(128, 3), (192, 3), (384, 3), (384, 20), (512, 3), (512, 10)])
@pytest.mark.parametrize("tv", [0, 1])
def test_default_kernel_resumes(H, S, tv):
    """Steps of 5 from the stored state (at 384 p lies in chi_out, at 384 and 512 the row slots lie in the
    chibar scratch), also with more slices than clusters: bit for bit the straight solve."""
    field, mask, _ = problem(H, S)
    assert np.array_equal(solve(field, mask, every=5, tv=tv), solve(field, mask, kernel=pcs.KERNEL_STREAMING, tv=tv))


@pytest.mark.parametrize("H", [64, 192, 256, 384])
@pytest.mark.parametrize("lam", [1e-5, 100.0])
def test_default_kernel_over_lambda(H, lam):
    """Beyond both ends of the scale that brings W p to the size of chi (16 .. 65536)."""
    field, mask, _ = problem(H, 2)
    check(solve(field, mask, lam=lam), field, mask, lam=lam)
