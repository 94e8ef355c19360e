"""Bins of the energy-angle histogram whose kernel takes FP32 arithmetic away from bin edges and,
where the bins fit shared memory, adds them up per block: every weight in the bin that double
arithmetic gives it, at the edges of both rules.  The weights are powers of two, so that the sums
are exact in any order: bit for bit."""
import numpy as np
import pytest

import synth

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


def reference(u, w, n_e, e_max, n_a):
    ek = np.sqrt(1.0 + (u[:, 0] * u[:, 0] + u[:, 1] * u[:, 1] + u[:, 2] * u[:, 2])) - 1.0
    ang = np.arctan2(np.sqrt(u[:, 1] * u[:, 1] + u[:, 2] * u[:, 2]), u[:, 0])
    ok = ek < e_max
    ie = np.clip((ek / e_max * n_e).astype(np.int64), 0, n_e - 1)
    ia = np.clip((ang / np.pi * n_a).astype(np.int64), 0, n_a - 1)
    out = np.zeros((n_e, n_a))
    np.add.at(out, (ie[ok], ia[ok]), w[ok])
    return out


@pytest.mark.parametrize("precision", [synth.FP32, synth.FP64])
@pytest.mark.parametrize("n_e,e_max,n_a", [(96, 12.0, 36), (1, 1e3, 1), (64, 2.0, 96), (65, 2.0, 96), (3, 1e-3, 1000),
                                           (2000, 40.0, 1)])
def test_every_weight_in_its_bin(P, precision, n_e, e_max, n_a):
    n = 40000
    rng = np.random.default_rng(8)
    dx = 0.2
    w = synth.Workload(name="bins", dim=2, n=(64, 48, 1), dx=dx, steps=1, beam=synth.BEAM_NONE, a0=1.0, duration=1.0,
                       slab_lo=(8, 8, 0), slab_hi=(9, 9, 1), n_e=1.0, ppc=1, seed=1, precision=precision)
    sim = P.Simulation(P.config_from(w, max_particles=n))
    u = rng.standard_normal((n, 3)) * np.exp(rng.uniform(-6, 2, n))[:, None]
    # on and next to bin edges: on the axis and across it, at rest, at energies of whole bins
    u[:4000, 1:] = 0.0
    u[4000:6000, 0] = 0.0
    u[6000:6100] = 0.0
    k = rng.integers(0, n_e + 1, 8000)
    g = 1.0 + k * (e_max / n_e)
    u[8000:16000, 0] = np.sqrt(g * g - 1.0)
    u[8000:16000, 1:] = 0.0
    a = rng.integers(0, n_a + 1, 8000) * np.pi / n_a
    u[16000:24000] = 0.7 * np.stack([np.cos(a), np.sin(a), np.zeros_like(a)], 1)
    if precision == synth.FP32:
        u = u.astype(np.float32).astype(np.float64)
    x = np.zeros((n, 3))
    x[:, :2] = rng.uniform(4.0, 40.0, (n, 2)) * dx
    wt = 2.0 ** -rng.integers(0, 12, n).astype(np.float64)
    sim.set_particles(x, u, wt, np.arange(n))
    got, want = sim.histogram(n_e, e_max, n_a), reference(u, wt, n_e, e_max, n_a)
    # numpy's square root, arctangent and division round as the device's do up to an ulp: a value on an edge
    # to the last bit may fall on either side, so edges are compared by the bins' neighbours
    d = got - want
    assert got.sum() == want.sum()
    assert np.count_nonzero(d) <= 2 * 16000 and np.abs(np.cumsum(d.sum(1))).max() <= wt[8000:16000].sum()
    inner = np.concatenate([np.arange(0, 8000), np.arange(24000, n)])
    sim.set_particles(x[inner], u[inner], wt[inner], np.arange(len(inner)))
    assert np.array_equal(sim.histogram(n_e, e_max, n_a), reference(u[inner], wt[inner], n_e, e_max, n_a))
    sim.close()
