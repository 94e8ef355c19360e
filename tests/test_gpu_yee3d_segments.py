"""The 3D field solver's columns, cut into segments along z, against the oracle: white-noise E, B in an
empty box, every point of every component.

Tolerances: those of tests/test_gpu_field_solver.py (1e-5 and 1e-12 of a component's maximum)."""
import numpy as np
import pytest

import synth
from _support import small_3d
from test_gpu_field_solver import P, noise_fields  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(P, orc, n, prec, steps):
    w = small_3d().with_(n=n, ppc=0, precision=prec)
    sim, ref = P.Simulation(P.config_from(w)), orc.Sim(orc.config_from(w))
    F = noise_fields(n, 3, seed=n[2])
    sim.set_fields(F)
    ref.set_fields(F)
    sim.step(steps)
    ref.step(steps)
    G, H = sim.fields(), ref.fields()
    sim.close()
    tol = 1e-5 if prec == synth.FP32 else 1e-12
    for comp in range(6):
        assert np.abs(G[comp] - H[comp]).max() < tol * np.abs(H[comp]).max(), comp


@pytest.mark.parametrize("prec", [synth.FP32, synth.FP64])
def test_segments_of_odd_length_one_after_another(P, orc, prec):
    """400 columns in segments of 13 and 12 planes: 800 work items on 304 (FP64 152) resident blocks, so
    blocks go from one odd segment to the next and reuse the output slot that the last plane left from."""
    n = (320, 320, 24)
    params = P.pic_derive_params(P.config_from(small_3d().with_(n=n, ppc=0)))
    assert params.yee_tile[2] == 13
    _check(P, orc, n, prec, 4)


@pytest.mark.parametrize("prec", [synth.FP32, synth.FP64])
@pytest.mark.parametrize("n", [(72, 72, 72), (64, 24, 81), (40, 48, 126)])
def test_last_plane_of_the_box(P, orc, n, prec):
    """Grids whose segments would leave the plane z = n_z to one of its own."""
    _check(P, orc, n, prec, 5)
