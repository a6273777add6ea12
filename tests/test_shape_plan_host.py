"""The cluster shape a call without variant options takes, chosen on the host."""

import os
import shutil

import pytest

import paper_2006_09808_gb300 as pcs

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists(pcs.LIB_PATH),
                                reason="needs nvcc or a built libpcs.so")

# resident clusters by cluster size, as a 152-SM device reports them
RESIDENT = {64: {4: 37, 2: 76, 1: 152}, 128: {8: 19, 4: 36, 2: 76, 1: 152}, 192: {12: 8, 6: 20, 3: 48},
            256: {16: 8, 8: 15, 4: 36}, 384: {8: 15}, 512: {16: 8}}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2006_09808_gb300 import build

    build.build()


def plan(H, S, **query):
    return pcs.pcs_shape_plan(H, H, S, RESIDENT[H], **query)


@pytest.mark.parametrize("H,S,balanced,whole", [
    # one slice more than the larger clusters hold: a fraction of a round on the balanced schedule,
    # a whole round without it
    (128, 19, 8, 8), (128, 21, None, 4), (192, 8, 12, 12), (192, 9, 12, 6), (256, 8, 16, 16), (256, 9, 16, 8),
    (256, 15, 8, 8), (256, 16, 8, 4), (256, 37, 4, 4),
])
def test_whole_slices_cost_whole_rounds(H, S, balanced, whole):
    if balanced:
        assert plan(H, S) == (balanced, min(S, RESIDENT[H][balanced]))
    assert plan(H, S, whole_slices=1) == (whole, min(S, RESIDENT[H][whole]))


def test_arguments():
    for H in RESIDENT:
        c, k = plan(H, 1)
        assert c == max(RESIDENT[H]) and k == 1  # a slice alone takes the largest cluster
    with pytest.raises(pcs.PcsError):
        plan(256, 0)
    with pytest.raises(pcs.PcsError):
        pcs.pcs_shape_plan(100, 100, 1, {4: 1})
