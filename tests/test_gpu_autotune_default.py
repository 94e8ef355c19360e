"""The autotuner always tries the default tile: what it picks for a large run of few electrons per cell, whose
small tiles it otherwise leaves out, is at least as fast as the default, within the trials' noise.

Bar: 6 %, between the noise of a trial (the better of two runs; a few per cent on a shared GPU, and a later
candidate replaces the first only by more than 1 %) and what tiles of 8x8x8 cost here (0.299 against 0.267
ms a step, 12 %), with which the search came out when it took those for the default."""
import pytest

import synth
from _support import small_3d
from test_gpu_field_solver import P  # noqa: F401

pytestmark = pytest.mark.gpu


def test_default_tile_is_tried(P):
    n = (112, 112, 112)
    w = small_3d().with_(n=n, slab_lo=(9, 9, 9), slab_hi=(103, 103, 103), ppc=2,
                         focus=tuple(0.5 * m * small_3d().dx for m in n))
    open_, fixed = P.config_from(w), P.config_from(w)
    default = list(P.pic_derive_params(P.config_from(w)).tile)
    for d in range(3):
        fixed.tile[d] = default[d]
    ms_fixed, ms_open = P.pic_autotune(fixed, 6), P.pic_autotune(open_, 6)
    assert ms_open <= 1.06 * ms_fixed, (list(open_.tile), ms_open, default, ms_fixed)
