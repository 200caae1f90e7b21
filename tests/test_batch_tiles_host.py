"""Which form the grids of a batch run in: marching strips or shared-memory tiles (host rule, no GPU).

A marching tile is one or two strips of 4 (32 - 2t) columns; a shared-memory tile's width is a power of two.
"""
import pytest

from paper_2603_00477_gb300 import binding as B
from paper_2603_00477_gb300 import build as gbuild
from paper_2603_00477_gb300 import inputs


@pytest.fixture(scope="module", autouse=True)
def lib():
    gbuild.build()
    B.load()


def marches(kinds, n, side, t, dtype="f32"):
    grids = []
    for i in range(n):
        shape, r = kinds[i % len(kinds)]
        grids.append((shape, r, side, side, inputs.weights(shape, 2, r, i)))
    b = B.Batch(grids, dtype, t)
    out = []
    for i in range(n):
        info = b.info(i)
        cw = 4 * (32 - 2 * info["t"])
        out.append(info["tile"][2] in (cw, 2 * cw))
    b.close()
    return out


# a small batch of long items leaves the chip idle when it marches; short items and larger batches march
@pytest.mark.parametrize("kind,n,side,t,march", [
    (("box", 3), 16, 64, 1, False), (("box", 3), 1, 64, 1, False), (("box", 2), 16, 64, 2, False),
    (("star", 3), 16, 90, 2, False), (("box", 2), 16, 90, 1, False), (("star", 2), 16, 90, 2, False),
    (("star", 1), 16, 90, 2, True), (("box", 1), 16, 90, 1, True), (("box", 2), 4, 64, 1, True),
    (("box", 3), 1, 1200, 1, False), (("box", 3), 16, 130, 1, True), (("star", 3), 30, 500, 2, True)])
def test_small_batches_of_long_items_stage(kind, n, side, t, march):
    assert marches([kind], n, side, t) == [march] * n


def test_depths_without_a_marching_kernel_stage():
    assert not any(marches([("star", 3)], 30, 500, 3))
    assert not any(marches([("box", 3)], 30, 500, 2))
    assert not any(marches([("box", 1)], 30, 500, 1, "f64"))


@pytest.mark.parametrize("others,march", [(3, True), (5, False)])
def test_mixed_batches_follow_the_larger_part(others, march):
    """Box-2D3R has no marching kernel at t = 2: where its grids hold about half of the points, all grids stage."""
    kinds = [("star", 2)] * (10 - others) + [("box", 3)] * others
    got = marches(kinds, 10, 300, 2)
    assert got == [march and k[0] == "star" for k in kinds]


def test_a_single_grid_takes_items_of_one_round():
    """1200 x 1200, Box-2D2R: eight rows per warp (190 items on 304 resident CTAs), not four (375: two rounds)."""
    b = B.Batch([("box", 2, 1200, 1200, inputs.weights("box", 2, 2, 1))], "f32", 1)
    assert b.info(0)["tile"][1:] == [32, 240]
    b.close()
