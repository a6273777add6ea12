"""The cluster shape a call without variant options takes, chosen on the host."""

import os
import shutil

import pytest

import paper_2006_09808_gb300 as pcs

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists(pcs.LIB_PATH),
                                reason="needs nvcc or a built libpcs.so")

# resident clusters by cluster size, as a 152-SM device reports them
RESIDENT = {64: {4: 76, 2: 152, 1: 152}, 128: {8: 38, 4: 36, 2: 76, 1: 152}, 192: {12: 23, 6: 23, 3: 48},
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
    (64, 38, 4, 4), (64, 39, 2, 2), (128, 19, 8, 8), (128, 20, 4, 4), (192, 12, 12, 12),
    (192, 16, 6, 6), (192, 24, 6, 3), (256, 8, 16, 16), (256, 9, 16, 8), (256, 15, 8, 8), (256, 19, 8, 4),
    (256, 20, 4, 4), (256, 37, 4, 4),
])
def test_whole_slices_cost_whole_rounds(H, S, balanced, whole):
    assert plan(H, S) == (balanced, min(S, RESIDENT[H][balanced]))
    assert plan(H, S, whole_slices=1) == (whole, min(S, RESIDENT[H][whole]))


@pytest.mark.parametrize("H,base", [(64, 1), (128, 4), (192, 2), (256, 4), (384, 4), (512, 8)])
def test_max_clusters_bounds_the_sms(H, base):
    """At most max_clusters clusters on at most that many times the base's SMs; only the smallest shape rounds up."""
    least = min(c for c in RESIDENT[H] if H != 128 or c > 1)  # 128's one-CTA shape is by option only
    for cap in (1, 2, 3, 5, 8, 16, 36, 200):
        for S in (1, 2, 7, 20, 64):
            for whole in (0, 1):
                c, k = plan(H, S, max_clusters=cap, whole_slices=whole)
                assert 1 <= k <= min(cap, S, RESIDENT[H][c])
                assert c * k <= cap * base or (c == least and c * (k - 1) < cap * base)
    assert plan(H, 64, max_clusters=1000) == plan(H, 64)


def test_max_clusters_choices():
    assert plan(256, 1, max_clusters=1) == (4, 1)
    assert plan(256, 1, max_clusters=4) == (16, 1)
    assert plan(256, 64, max_clusters=8) == (4, 8)
    assert plan(128, 64, max_clusters=8) == (4, 8)  # not 8 of the 2-CTA shape


@pytest.mark.parametrize("H,alone,crowd", [(64, 4, 1), (128, 8, 2), (192, 12, 3), (256, 16, 4)])
def test_solves_in_flight_shrink_the_clusters(H, alone, crowd):
    """Alone, a slice takes the largest cluster; beside many others the shape with the least SM time."""
    assert plan(H, 1)[0] == alone
    assert plan(H, 1, in_flight=200.0)[0] == crowd
    sizes = [plan(H, 1, in_flight=float(n))[0] for n in range(0, 200, 4)]
    assert sizes == sorted(sizes, reverse=True)
    assert plan(256, 1, solves=23, in_flight=23.0)[0] == 4  # 24 calls of one slice
    assert plan(192, 1, solves=31, in_flight=47.0)[0] == 3
    assert plan(192, 1, solves=35, in_flight=35.0)[0] < 12  # more streams than run at once: two solves in turn
    with pytest.raises(pcs.PcsError):
        plan(H, 1, in_flight=-1.0)


def test_device_without_room_for_the_chosen_shapes():
    """A part of a GPU that holds no 16-CTA (or 8-CTA) cluster solves with a half-spectrum variant."""
    assert pcs.pcs_shape_plan(512, 512, 5, {16: 0, 8: 2}) == (8, 2)
    assert pcs.pcs_shape_plan(512, 512, 5, {16: 1, 8: 2}, sms=15) == (8, 2)
    assert pcs.pcs_shape_plan(384, 384, 5, {8: 0, 4: 3}, max_clusters=2) == (4, 2)
    with pytest.raises(pcs.PcsError):
        pcs.pcs_shape_plan(512, 512, 5, {16: 0, 8: 0})


def test_arguments():
    for H in RESIDENT:
        c, k = plan(H, 1)
        assert c == max(RESIDENT[H]) and k == 1  # a slice alone takes the largest cluster
    with pytest.raises(pcs.PcsError):
        plan(256, 0)
    with pytest.raises(pcs.PcsError):
        pcs.pcs_shape_plan(100, 100, 1, {4: 1})
