"""Work items and the fixed-point current of the FP32 push where they can go wrong: default tiles
and work items at the edges of the rule that sizes them, and the largest sum one node can take
(every electron of the largest work items in one cell, moving together).

Tolerances.  Default items: the FP32 / FP64 bars of tests/_support.py.  The heavy node: each of
the N contributions to a node is rounded by at most half a unit of the fixed-point scale,
2^-30 max(N, 256) w, all the same way (the electrons are alike), so the sum by N times that; the
other FP32 operations of a contribution (some twenty roundings of 2^-24 each) add at most 20 2^-24
of the largest J."""
import numpy as np
import pytest

import synth
from _support import field_bar, field_errors, momentum_bar, momentum_error

pytestmark = pytest.mark.gpu
TWO_PI = 2 * np.pi


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_11393_gb300 import _build, pic

    _build.build()
    pic.load()
    return pic


def _slab(dim, n, ppc, precision):
    dx = TWO_PI / (32 if dim == 2 else 24)
    dt = 0.95 * dx / np.sqrt(dim)
    n = tuple(n) + (1,) * (3 - dim)
    return synth.Workload(name="items", dim=dim, n=n, dx=dx, steps=12, beam=synth.BEAM_LP, a0=8.0,
                          duration=synth.fs(5.0), w0=TWO_PI * 0.6,
                          slab_lo=tuple(4 if d < dim else 0 for d in range(3)),
                          slab_hi=tuple(n[d] - 5 if d < dim else 1 for d in range(3)), n_e=0.03, ppc=ppc, seed=5,
                          focus=tuple(0.5 * n[d] * dx if d < dim else 0.0 for d in range(3)), t_focus=6 * dt,
                          precision=precision)


@pytest.mark.parametrize("dim,n,ppc,precision", [
    (2, (61, 47), 1, synth.FP32),      # 256 electrons per 16x16 tile, item 256: tile 16x16
    (2, (33, 29), 7, synth.FP32),
    (2, (40, 40), 3, synth.FP64),
    (3, (17, 21, 23), 1, synth.FP32),  # one tile of 16 cells and one of 1
    (3, (33, 16, 19), 5, synth.FP32),
    (3, (18, 17, 20), 2, synth.FP64),
])
def test_default_tiles_and_items_match_the_oracle(P, orc, dim, n, ppc, precision):
    w = _slab(dim, n, ppc, precision)
    sim = P.Simulation(P.config_from(w))
    ref = orc.Sim(orc.config_from(w))
    sim.step(w.steps)
    ref.step(w.steps)
    pg, pr = sim.particles(), ref.particles()
    np.testing.assert_array_equal(np.sort(pg["id"]), np.sort(pr["id"]))
    prec = "fp32" if precision == synth.FP32 else "fp64"
    err, _ = momentum_error(pg, pr, w.a0, floor=1.0 if prec == "fp32" else 1e-3)
    assert err < (momentum_bar(w.steps, w.dt) if prec == "fp32" else 1e-9)
    assert field_errors(sim.fields(), ref.fields()).max() < field_bar(dim, w.steps, prec)
    sim.close()


@pytest.mark.parametrize("dim,tile", [(1, (32,)), (2, (16, 16)), (2, (40, 8)), (3, (16, 8, 4)), (3, (8, 8, 4)),
                                      (3, (20, 6, 5))])
@pytest.mark.parametrize("count,chunk", [(256, 256), (511, 512), (513, 1024), (16384, 16384)])
def test_every_electron_of_an_item_on_the_same_nodes(P, orc, dim, tile, count, chunk):
    dx = 0.2
    n = (32, 24, 20)[:dim] + (1,) * (3 - dim)
    w = synth.Workload(name="heavy", dim=dim, n=n, dx=dx, steps=1, beam=synth.BEAM_NONE, a0=1.0, duration=1.0,
                       slab_lo=(8,) * dim + (0,) * (3 - dim), slab_hi=(9,) * dim + (1,) * (3 - dim), n_e=1.0, ppc=1,
                       seed=1, precision=synth.FP32)
    sim = P.Simulation(P.config_from(w, tile=tile, chunk=chunk, max_particles=count))
    ref = orc.Sim(orc.config_from(w))
    # one cell corner to the next, nearly at the speed of light along +x, -y and +z
    x = np.zeros((count, 3))
    x[:, :dim] = (10 + 0.45) * dx
    u = np.zeros((count, 3))
    u[:] = np.array([60.0, -55.0, 50.0])
    wt = np.full(count, 0.7)
    ids = np.arange(count, dtype=np.int64)
    for s in (sim, ref):
        s.set_particles(x, u, wt, ids)
        s.step(1)
    Fg, Fr = sim.fields(), ref.fields()
    for c in range(6, 9):
        peak = np.abs(Fr[c]).max()
        assert peak > 0
        unit = 2.0**-30 * max(min(count, chunk), 256)
        bar = count * 0.7 * unit + 20 * 2.0**-24 * peak
        assert np.abs(Fg[c] - Fr[c]).max() < bar, (c, np.abs(Fg[c] - Fr[c]).max() / peak, bar / peak)
    sim.close()
