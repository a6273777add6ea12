"""The field map at the counts and alignments where its launches change: fewer voxels than the first
launch's CTAs, remainders of the two- and four-voxel steps, outputs aligned for two voxels only."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2006_09808_gb300 as pcs  # noqa: E402

pytestmark = pytest.mark.gpu
B0, T_SHIFT, THR = 3.0, 0.6e-3, 0.1


def run(s0, s1, offset):
    """Outputs start `offset` voxels into their buffers (2: 8- and 2-byte aligned only)."""
    n = s0.numel()
    f, w = (torch.full((n + 8,), float("nan"), device="cuda") for _ in range(2))
    m = torch.full((n + 8,), 77, dtype=torch.uint8, device="cuda")
    out = [t[offset:offset + n] for t in (f, w, m)]
    pcs.pcs_field_map(s0, s1, T_SHIFT, B0, THR, *out)
    torch.cuda.synchronize()
    assert bool(torch.isnan(f[offset + n:]).all()) and bool((m[offset + n:] == 77).all())  # nothing past the end
    assert bool((m[:offset] == 77).all())
    return [t.cpu().numpy().copy() for t in out]


@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 511, 512, 513, 514, 1027, 4099, 466945, 1000003])
def test_counts_and_alignments(n):
    rng = np.random.default_rng(n)
    z = (rng.standard_normal((2, n)) + 1j * rng.standard_normal((2, n))).astype(np.complex64)
    z[0, rng.integers(0, n)] *= 3.0  # the maximum anywhere, also among the first voxels
    s0, s1 = torch.from_numpy(z[0]).cuda(), torch.from_numpy(z[1]).cuda()
    field, weight, mask = run(s0, s1, 0)
    a, b = z[0].astype(np.complex128), z[1].astype(np.complex128)
    m2 = np.abs(a) ** 2
    near = np.abs(m2 - THR ** 2 * m2.max()) <= 1e-6 * m2.max() * THR ** 2  # float32 rounding of the cut
    ref = m2 >= THR ** 2 * m2.max()
    assert np.array_equal(mask[~near] != 0, ref[~near])
    rad = 2 * np.pi * 42.577478518 * B0 * T_SHIFT
    # the two products of each component cancel at worst to eps |a b|: an angle error of 4 eps
    err = np.angle(np.exp(1j * (field.astype(np.float64) * rad - np.angle(b * a.conj()))))
    assert np.all(np.abs(err[mask != 0]) <= 8 * 6e-8 + 4e-7) and np.all(field[mask == 0] == 0)
    assert np.allclose(weight, np.sqrt(m2 / m2.max()), rtol=0, atol=4e-7)
    for other in zip((field, weight, mask), run(s0, s1, 2)):
        assert np.array_equal(*other)
