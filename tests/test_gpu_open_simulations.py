"""Several simulations of different tiles open at once: what one opens or steps changes nothing for the
others.  The kernels are shared, their limits of shared memory with them.

Tolerances: the FP32 / FP64 bars of tests/_support.py against the oracle."""
import numpy as np
import pytest

import synth
from _support import field_bar, field_errors, momentum_bar, momentum_error, small_1d, small_2d, small_3d
from test_gpu_field_solver import P  # noqa: F401

pytestmark = pytest.mark.gpu

# (workload, tile of the simulation that steps, tile of the one opened after it): the second box is smaller, and
# both are pushed by the same kernel (1D; 2D and 3D FP32 boxes of one pitch; the general kernel)
PAIRS = [("1d", synth.FP64, (128,), (16,)), ("2d", synth.FP32, (32, 16), (32, 8)), ("2d", synth.FP64, (32, 32), (8, 8)),
         ("2d", synth.FP32, (48, 24), (20, 8)), ("3d", synth.FP32, (16, 8, 8), (16, 8, 4))]
MAKE = {"1d": small_1d, "2d": small_2d, "3d": small_3d}


@pytest.mark.parametrize("batch", [False, True], ids=["alone", "batch"])
@pytest.mark.parametrize("kind,precision,tile,other", PAIRS)
def test_many_steps_after_another_was_opened(P, orc, kind, precision, tile, other, batch):
    w = MAKE[kind]().with_(precision=precision)
    if kind == "3d":
        w = w.with_(a0=2.0)      # (its bars are measured up to 50 steps at a0 = 20)
    a = P.Simulation(P.config_from(w, tile=tile))
    b = P.Simulation(P.config_from(w, tile=other))
    if batch:                                          # a batch of the smaller ones sets the kernel up again
        c = P.Simulation(P.config_from(w.with_(seed=w.seed + 1), tile=other))
        P.pic_batch_step([b.h, c.h], 1)
        c.close()
    ref = orc.Sim(orc.config_from(w))
    a.step(64)
    ref.step(64)
    pa, pr = a.particles(), ref.particles()
    np.testing.assert_array_equal(np.sort(pa["id"]), np.sort(pr["id"]))
    assert len(pa["id"]) > 0
    prec = "fp32" if precision == synth.FP32 else "fp64"
    err, _ = momentum_error(pa, pr, w.a0, floor=1.0 if prec == "fp32" else 1e-3)
    assert err < (momentum_bar(64, w.dt) if prec == "fp32" else 1e-9)
    assert field_errors(a.fields(), ref.fields()).max() < field_bar(w.dim, 64, prec)
    seconds = P.pic_profile_step(a.h, 1)               # the kernels launched one by one, too
    assert (seconds >= 0).all() and a.info().step == 65
    a.close()
    b.close()
