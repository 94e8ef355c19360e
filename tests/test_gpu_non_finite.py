"""Values that are not finite: what the push and the incident field do with them, exactly (counts, ids,
NaN or not)."""
import numpy as np
import pytest

import synth
from _support import small_1d, small_2d, small_3d
from test_gpu_field_solver import P  # noqa: F401

pytestmark = pytest.mark.gpu

MAKE = {1: small_1d, 2: small_2d, 3: small_3d}


@pytest.mark.parametrize("dim", [1, 2, 3])
@pytest.mark.parametrize("axis", [0, 2])
def test_fp64_electron_of_no_momentum_is_removed(P, dim, axis):
    """A NaN momentum makes the move NaN, and the cell that a NaN converts to is outside the box."""
    w = MAKE[dim]().with_(precision=synth.FP64)
    sim = P.Simulation(P.config_from(w))
    p = sim.particles()
    n = len(p["id"])
    u, lost = p["u"].copy(), p["id"][n // 2]
    u[n // 2, axis] = np.nan
    sim.set_particles(p["x"], u, p["w"], p["id"])
    sim.step(1)
    assert sim.info().n_alive == n - 1 and sim.info().n_exits == 1
    assert lost not in sim.particles()["id"] and sim.exits()["id"][0] == lost
    sim.close()


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("beam", [synth.BEAM_LP, synth.BEAM_RP])
@pytest.mark.parametrize("precision", [synth.FP32, synth.FP64])
def test_incident_field_where_a_coordinate_is_no_number(P, dim, beam, precision):
    """NaN in, NaN out, as the closed form's formulas give: not a field of zero."""
    w = MAKE[dim]().with_(beam=beam, precision=precision, ppc=0)
    sim = P.Simulation(P.config_from(w))
    at = np.array([*w.focus, w.t_focus])
    pts = np.tile(at + 0.3 * w.dx, (6, 1))
    for k, d in enumerate([0, 1, 3] if dim == 2 else [0, 1, 2, 3]):
        pts[k, d] = np.nan
    out = sim.eval_incident(pts)
    bad = np.isnan(pts).any(1)
    assert np.isnan(out[bad]).any(1).all()
    assert np.isfinite(out[~bad]).all() and (out[~bad] != 0).any(1).all()
    sim.close()


def test_energies_far_from_a_tiny_focus(P):
    """A confocal parameter so small that |u|^2 of the closed form leaves single precision: finite."""
    w = MAKE[3]().with_(a_param=1e-9, ppc=0)
    sim = P.Simulation(P.config_from(w))
    assert np.isfinite(sim.energies()).all()
    sim.close()
