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
