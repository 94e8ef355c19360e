"""Particle tiles that a configuration leaves open, from pic_derive_params (host only)."""
import pytest

import synth
from _support import small_1d, small_2d, small_3d


@pytest.fixture(scope="module")
def P():
    from paper_2310_11393_gb300 import _build, pic

    _build.build()
    pic.load()
    return pic


CASES = [(small_1d, (0,), (32, 1, 1)), (small_2d, (0, 0), (16, 16, 1)), (small_2d, (32, 0), (32, 16, 1)),
         (small_2d, (0, 8), (16, 8, 1)),
         (small_3d, (0, 0, 0), (16, 8, 4)), (small_3d, (0, 0, 16), (8, 8, 16)), (small_3d, (0, 16, 8), (8, 16, 8)),
         (small_3d, (0, 0, 8), (8, 8, 8)), (small_3d, (32, 0, 2), (32, 8, 2)), (small_3d, (16, 8, 8), (16, 8, 8))]


@pytest.mark.parametrize("precision", [synth.FP32, synth.FP64])
@pytest.mark.parametrize("make,given,want", CASES)
def test_open_axes(P, make, given, want, precision):
    """All axes open: the default tile.  Some given: 8 cells (2D 16) along the others, so that boxes that fit the
    shared memory go on fitting it (16 x 16 x 8 cells in FP32 and 16 x 8 x 8 in FP64 would not)."""
    cfg = P.config_from(make().with_(precision=precision))
    for d, t in enumerate(given):
        cfg.tile[d] = t
    assert tuple(P.pic_derive_params(cfg).tile) == want
