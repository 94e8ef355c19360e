"""3D simulations whose configuration sets the particle tile along some axes only: opened (their boxes fit
the shared memory) and stepped, against the oracle at the bars of tests/_support.py."""
import pytest

import synth
from _support import field_bar, field_errors, momentum_bar, momentum_error, small_3d
from test_gpu_field_solver import P  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tile", [(synth.FP32, (0, 0, 16)), (synth.FP32, (0, 16, 8)), (synth.FP64, (0, 0, 8))])
def test_tile_along_some_axes(P, orc, precision, tile):
    w = small_3d(precision=precision)
    cfg = P.config_from(w)
    for d in range(3):
        cfg.tile[d] = tile[d]
    sim, ref = P.Simulation(cfg), orc.Sim(orc.config_from(w))
    sim.step(10)
    ref.step(10)
    prec = "fp32" if precision == synth.FP32 else "fp64"
    err, n = momentum_error(sim.particles(), ref.particles(), w.a0, floor=1.0 if prec == "fp32" else 1e-3)
    assert n > 0 and err < (momentum_bar(10, w.dt) if prec == "fp32" else 1e-9)
    assert field_errors(sim.fields(), ref.fields()).max() < field_bar(3, 10, prec)
    sim.close()
