"""Segments of the 3D field solver's columns, from pic_derive_params (host only).  A segment evaluates
the Mur condition of the face z = n_z from E on the plane before, which it has only if that plane is its
own: no segment may start on plane n_z."""
import pytest

from _support import small_3d


@pytest.fixture(scope="module")
def P():
    from paper_2310_11393_gb300 import _build, pic

    _build.build()
    pic.load()
    return pic


def test_no_segment_starts_on_the_last_plane(P):
    grids = [(n, n, n) for n in range(16, 260)] + [(64, 64, n) for n in range(16, 600, 3)] + [(512, 256, 256), (96, 96, 132)]
    for n in grids:
        w = small_3d().with_(n=n, ppc=0)
        yt = P.pic_derive_params(P.config_from(w)).yee_tile[2]
        last = n[2] + 1 - (n[2] // yt) * yt          # planes of the last of ceil((n_z + 1) / yt) segments
        assert yt >= 8 and (last >= 2 or yt > n[2]), (n, yt)
        assert yt <= 65, (n, yt)
