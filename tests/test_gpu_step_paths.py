"""The routes of a step and of the state's input and output: many steps in one graph launch, the tile
scan on the field solver's launch and in one of its own, particles and fields through
more pieces than fit the staging memory at once.

Tolerances.  Steps: the FP32 / FP64 bars of tests/_support.py against the oracle.  Input and output: a
position is kept as a cell and an offset in it, so it comes back within two roundings of the offset
in cells and two of the product with dx (4 units of its size in FP64); everything else is kept as
given."""
import numpy as np
import pytest

import synth
from _support import field_bar, field_errors, momentum_bar, momentum_error, small_2d

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_11393_gb300 import _build, pic

    _build.build()
    pic.load()
    return pic


def _compare(sim, ref, w, steps, prec):
    pg, pr = sim.particles(), ref.particles()
    np.testing.assert_array_equal(np.sort(pg["id"]), np.sort(pr["id"]))
    err, _ = momentum_error(pg, pr, w.a0, floor=1.0 if prec == "fp32" else 1e-3)
    assert err < (momentum_bar(steps, w.dt) if prec == "fp32" else 1e-9)
    assert field_errors(sim.fields(), ref.fields()).max() < field_bar(w.dim, steps, prec)


@pytest.mark.parametrize("calls", [(64,), (79,), (3, 64, 1, 12), (63,)])
@pytest.mark.parametrize("sort_every,ppc", [(0, 4), (5, 4), (5, 8)])     # (lane strides 1, 4, 4 of 128 threads)
def test_many_steps_in_one_call(P, orc, calls, sort_every, ppc):
    w = small_2d(precision=synth.FP64).with_(ppc=ppc)
    sim = P.Simulation(P.config_from(w, sort_every=sort_every))
    ref = orc.Sim(orc.config_from(w))
    for n in calls:
        sim.step(n)
    ref.step(sum(calls))
    assert sim.info().step == sum(calls)
    _compare(sim, ref, w, sum(calls), "fp64")
    sim.close()


@pytest.mark.parametrize("n,tile", [((256, 256, 1), (4, 4)), ((257, 256, 1), (4, 4)),        # 4096, 4160 tiles
                                    ((1040, 1025, 1), (16, 16)), ((1040, 1025, 1), (8, 8))])  # 4225, 16770 tiles
@pytest.mark.parametrize("precision", [synth.FP32, synth.FP64])
def test_tile_scan_with_and_beside_the_field_solver(P, orc, n, tile, precision):
    w = small_2d(precision=precision, steps=20).with_(n=n, slab_hi=(n[0] - 4, 100, 1), ppc=1)
    sim = P.Simulation(P.config_from(w, tile=tile))
    ref = orc.Sim(orc.config_from(w))
    sim.step(w.steps)
    ref.step(w.steps)
    _compare(sim, ref, w, w.steps, "fp32" if precision == synth.FP32 else "fp64")
    sim.close()


def _electrons(w, n, seed):
    rng = np.random.default_rng(seed)
    x = np.zeros((n, 3))
    for d in range(w.dim):
        x[:, d] = rng.uniform(8.0, w.n[d] - 8.0, n) * w.dx
    return x, rng.normal(size=(n, 3)), rng.uniform(0.5, 1.0, n), rng.permutation(n)


@pytest.mark.parametrize("n", [1, 1 << 20, (1 << 20) + 1, 2500003])
def test_particles_through_the_staging_memory(P, n):
    w = small_2d(precision=synth.FP64).with_(ppc=1)
    sim = P.Simulation(P.config_from(w, max_particles=2500003))
    x, u, wt, ids = _electrons(w, n, 3)
    sim.set_particles(x, u, wt, ids)
    p = sim.particles()
    assert len(p["id"]) == n
    o, q = np.argsort(p["id"]), np.argsort(ids)
    np.testing.assert_array_equal(p["id"][o], ids[q])
    np.testing.assert_array_equal(p["u"][o], u[q])
    np.testing.assert_array_equal(p["w"][o], wt[q])
    assert (np.abs(p["x"][o] - x[q]) <= 4 * 2.0**-53 * np.abs(x[q]).max()).all()
    # a particle outside, in the last piece: refused, and nothing changed
    bad = x.copy()
    bad[-1, 1] = -1.0
    with pytest.raises(P.PicError):
        sim.set_particles(bad, 2 * u, wt, ids)
    again = sim.particles()
    for k in ("x", "u", "w", "id"):
        np.testing.assert_array_equal(again[k], p[k])
    sim.close()


@pytest.mark.parametrize("precision", [synth.FP32, synth.FP64])
@pytest.mark.parametrize("n,ppc", [((300, 200, 1), 1), ((40, 40, 1), 64)])     # one component a piece; all at once
def test_fields_through_the_staging_memory(P, n, ppc, precision):
    w = small_2d(precision=precision).with_(n=n, slab_lo=(16, 16, 0), slab_hi=(24, 24, 1), ppc=ppc)
    sim = P.Simulation(P.config_from(w))
    F = np.random.default_rng(4).normal(size=(9, 1, n[1] + 1, n[0] + 1)).astype(np.float32).astype(np.float64)
    before = sim.fields()
    sim.set_fields(F)
    got = sim.fields()
    np.testing.assert_array_equal(got[6:], before[6:])
    inner = (slice(0, 6), slice(None), slice(0, n[1]), slice(0, n[0]))
    np.testing.assert_array_equal(got[inner], F[inner])
    sim.close()
