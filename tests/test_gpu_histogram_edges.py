"""Bins of the energy-angle histogram for momenta on and next to bin edges, one electron at a time.

Every electron of a call has a weight of its own power of two, so the bins say where each one went.
The admissible bins come from the energy and the angle in extended precision, widened by the rounding
of double arithmetic: gamma - 1 carries four roundings of gamma's size, the quotients two more; the
angle four of its own (a square root, two products, an arctangent of one unit) and two of the quotient.
So an electron a single-precision unit away from an edge has one admissible bin, and one within those
few double-precision units of it two."""
import numpy as np
import pytest

import synth
from test_gpu_field_solver import P  # noqa: F401

pytestmark = pytest.mark.gpu

L = np.longdouble
EPS = L(2.0) ** -53


def admissible(u, n_e, e_max, n_a):
    """(energy bins, angle bins) of each momentum; energy bin n_e: not counted."""
    u = u.astype(L)
    up = u[:, 1] ** 2 + u[:, 2] ** 2
    u2 = u[:, 0] ** 2 + up
    gamma = np.sqrt(1 + u2)
    e = u2 / (1 + gamma)
    te, de = e / L(e_max) * n_e, (4 * gamma + 4 * e) * EPS / L(e_max) * n_e
    ta = np.arctan2(np.sqrt(up), u[:, 0]) / (4 * np.arctan(L(1))) * n_a
    da = 8 * ta * EPS
    out = []
    for t, d, n in ((te, de, n_e), (ta, da, n_a - 1)):
        out.append(np.stack([np.clip(np.floor(t - d), 0, n), np.clip(np.floor(t + d), 0, n)], 1).astype(int))
    return out


def momenta(n_e, e_max, n_a, rng):
    """Single-precision momenta on the edges of up to 200 bins of each axis and up to four units either side."""
    kind = np.float32
    k = np.unique(rng.integers(0, n_e + 1, 200))
    g = 1.0 + k * (e_max / n_e)
    rows = [np.stack([s * np.sqrt(g * g - 1.0) * (g > 1), 0 * g, 0 * g], 1) for s in (1, -1)]
    a = np.unique(rng.integers(0, n_a + 1, 200)) * np.pi / n_a
    for r in (0.7, 1e-4, 30.0):
        rows.append(r * np.stack([np.cos(a), np.sin(a), 0 * a], 1))
        rows.append(r * np.stack([np.cos(a), 0.6 * np.sin(a), 0.8 * np.sin(a)], 1))
    u = np.concatenate(rows).astype(kind)
    out = [u]
    for axis in range(2):
        for way in (-1, 1):
            v = u.copy()
            for _ in range(4):
                step = np.nextafter(v[:, axis], kind(way * np.inf))
                v[:, axis] = np.where(v[:, axis] == 0, 0, step)      # (what is on the axis stays there)
                out.append(v.copy())
    return np.unique(np.concatenate(out), axis=0).astype(np.float64)


@pytest.mark.parametrize("shared", [False, True], ids=["global_bins", "shared_bins"])
@pytest.mark.parametrize("precision", [synth.FP32, synth.FP64])
@pytest.mark.parametrize("n_e,e_max,n_a", [(96, 12.0, 36), (64, 2.0, 90), (3, 1e-3, 700)])
def test_every_electron_in_an_admissible_bin(P, precision, n_e, e_max, n_a, shared):
    group = 48                                            # powers of two that a double sums exactly
    fill = 16 * n_e * n_a if shared else 0                # electrons of no weight: enough for bins in shared memory
    dx = 0.2
    w = synth.Workload(name="edges", dim=2, n=(64, 48, 1), dx=dx, steps=1, beam=synth.BEAM_NONE, a0=1.0, duration=1.0,
                       slab_lo=(8, 8, 0), slab_hi=(9, 9, 1), n_e=1.0, ppc=1, seed=1, precision=precision)
    sim = P.Simulation(P.config_from(w, max_particles=group + fill))
    rng = np.random.default_rng(n_e)
    us = momenta(n_e, e_max, n_a, rng)
    us = us[rng.permutation(len(us))[:1920]]
    both = 0
    for i in range(0, len(us), group):
        u = us[i:i + group]
        ae, aa = admissible(u, n_e, e_max, n_a)
        m = len(u)
        n = m + fill
        x = np.zeros((n, 3))
        x[:, :2] = rng.uniform(4.0, 40.0, (n, 2)) * dx
        wt = np.zeros(n)
        wt[:m] = 2.0 ** (np.arange(m) - 24)
        sim.set_particles(x, np.concatenate([u, np.zeros((fill, 3))]), wt, np.arange(n))
        H = sim.histogram(n_e, e_max, n_a)
        bits = (H * 2.0**24).astype(np.int64)
        np.testing.assert_array_equal(bits, H * 2.0**24)
        for j in range(m):
            got = np.argwhere((bits >> j) & 1)
            both += int(ae[j, 0] != ae[j, 1] or aa[j, 0] != aa[j, 1])
            if len(got) == 0:
                assert ae[j, 1] == n_e, (u[j], ae[j])
                continue
            assert len(got) == 1 and ae[j, 0] <= got[0, 0] <= ae[j, 1] and aa[j, 0] <= got[0, 1] <= aa[j, 1], \
                (u[j].tolist(), got.tolist(), ae[j], aa[j])
    assert both < 0.1 * len(us)                           # (nearly all have one bin only)
    sim.close()


@pytest.mark.parametrize("precision", [synth.FP32, synth.FP64])
def test_energies_at_the_rounding_of_gamma(P, precision):
    """gamma - 1 in double has steps of 2.2e-16, whatever the precision of the run: a spectrum up to 1e-14
    has them in its bins.  Momenta at 45 degrees, whose squares and their sum are exact in double: exact."""
    n, n_e, e_max = 20000, 50, 1e-14
    dx = 0.2
    w = synth.Workload(name="edges", dim=2, n=(64, 48, 1), dx=dx, steps=1, beam=synth.BEAM_NONE, a0=1.0, duration=1.0,
                       slab_lo=(8, 8, 0), slab_hi=(9, 9, 1), n_e=1.0, ppc=1, seed=1, precision=precision)
    sim = P.Simulation(P.config_from(w, max_particles=n))
    rng = np.random.default_rng(2)
    x, u = np.zeros((n, 3)), np.zeros((n, 3))
    x[:, :2] = rng.uniform(4.0, 40.0, (n, 2)) * dx
    u[:, 0] = u[:, 1] = np.exp(rng.uniform(np.log(1e-9), np.log(1.4e-7), n)).astype(np.float32)
    ek = np.sqrt(1.0 + 2.0 * (u[:, 0] * u[:, 0])) - 1.0
    want = np.bincount((ek[ek < e_max] / e_max * n_e).astype(int), minlength=n_e)
    sim.set_particles(x, u, np.ones(n), np.arange(n))
    np.testing.assert_array_equal(sim.histogram(n_e, e_max, 1)[:, 0], want)
    sim.close()
