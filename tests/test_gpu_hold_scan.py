"""pic_test_hold_scan where one block of the field solver's launch scans the tiles (4097 to 16384 of them, of
256 cells): the wait runs out and is reported as for larger runs, and steps go on as before with
publishing restored (FP64 bar of tests/_support.py).  Bounded waits; no TMA copy is
pending during them."""
import pytest

import synth
from _support import field_errors, momentum_error, small_2d
from test_gpu_field_solver import P  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture
def workload():
    return small_2d(precision=synth.FP64).with_(n=(1040, 1025, 1), slab_hi=(1036, 100, 1), ppc=1)   # 4225 tiles of 16 x 16


def test_wait_that_runs_out_is_reported(P, workload):
    sim = P.Simulation(P.config_from(workload))
    sim.step(1)
    assert sim.info().status == 0
    P.pic_test_hold_scan(sim.h, 0, 1 << 12)
    sim.step(1)
    assert sim.info().status & P.PIC_FLAG_TIMEOUT
    with pytest.raises(P.PicError) as e:
        sim.energies()
    assert e.value.status == P.PIC_ETIMEOUT
    sim.close()


def test_steps_go_on_after_it(P, orc, workload):
    sim, ref = P.Simulation(P.config_from(workload)), orc.Sim(orc.config_from(workload))
    sim.step(3)
    P.pic_test_hold_scan(sim.h, -1, 1 << 22)
    sim.step(3)
    ref.step(6)
    assert sim.info().status == 0 and sim.info().step == 6
    err, n = momentum_error(sim.particles(), ref.particles(), workload.a0, floor=1e-3)
    assert n > 0 and err < 1e-9 and field_errors(sim.fields(), ref.fields()).max() < 1e-9
    sim.close()
