"""The FP32 current of the 3D push, bit for bit: Esirkepov's sum in the order and with the roundings that
push.cu states, in numpy, against the GPU for electrons of one work item.

Exact (no tolerance): the electrons move freely with 1 + u^2 = 4 to the last bit, so that the velocity is
u/2 whatever the inverse square root rounds; those are taken whose new offset is the same with one
rounding or two; every other operation of the deposit is one IEEE operation.  The sums are integers,
in any order."""
import numpy as np
import pytest

import synth
from _support import small_3d
from test_gpu_field_solver import P  # noqa: F401

pytestmark = pytest.mark.gpu
F = np.float32


def fma(a, b, c):
    """One rounding (the double product of floats is exact)."""
    return (a.astype(np.float64) * np.asarray(b, np.float64) + np.asarray(c, np.float64)).astype(F)


def shape(d):
    return [F(0.5) * (F(0.5) - d) * (F(0.5) - d), fma(-d, d, F(0.75)), F(0.5) * (F(0.5) + d) * (F(0.5) + d)]


def momenta(n, rng):
    """u with 1 + u^2 = 4 in single precision for every order of the sum and with or without FMAs."""
    out = np.zeros((0, 3), F)
    while len(out) < n:
        u = rng.normal(size=(4 * n, 3))
        u = (u * np.sqrt(3.0 / (u * u).sum(1))[:, None]).astype(F)
        ok = np.ones(len(u), bool)
        for i, j, k in ((0, 1, 2), (1, 0, 2), (2, 1, 0), (0, 2, 1), (1, 2, 0), (2, 0, 1)):
            a, b, c = u[:, i], u[:, j], u[:, k]
            plain = (a * a + b * b) + c * c
            for s in (F(1) + plain, F(1) + fma(c, c, fma(b, b, a * a)), fma(c, c, fma(b, b, fma(a, a, F(1))))):
                ok &= s == F(4)
        out = np.concatenate([out, u[ok]])
    out[:8] = [[(1, -1)[(k >> d) & 1] for d in range(3)] for k in range(8)]
    return out[:n]


def current(cell, o, u, wt, n, dx, dt, items):
    """Integer units of J[3][z][y][x] that the electrons add."""
    wmax = np.nextafter(F(wt.max()), F(np.inf))
    q = F(536870912.0) / (F(items) * wmax)
    dtdx, cw = F(dt * (1.0 / dx)), F(dx / dt) * wt
    S, D, base = [], [], []
    for d in range(3):
        h = (o[:, d] >= F(0.5)).astype(F)
        d0 = o[:, d] - h
        r1 = d0 + dtdx * (u[:, d] * F(0.5))
        sh = np.floor(r1 + F(0.5))
        w0, w1 = shape(d0), shape(r1 - sh)
        lo, hi, z = sh < 0, sh > 0, np.zeros_like(d0)
        old = [np.where(lo, z, w0[0]), np.where(lo, w0[0], w0[1]), np.where(lo, w0[1], w0[2]), np.where(lo, w0[2], z)]
        new = [np.where(hi, z, w1[0]), np.where(hi, w1[0], w1[1]), np.where(hi, w1[1], w1[2]), np.where(hi, w1[2], z)]
        S.append(old)
        D.append([b - a for a, b in zip(old, new)])
        base.append(cell[:, d] + h.astype(int) - 1 - lo)
    J = np.zeros((3, n[2] + 1, n[1] + 1, n[0] + 1), np.int64)
    third = F(1) / F(3)
    for d in range(3):
        t, z = (1, 2) if d == 0 else (0, 2) if d == 1 else (0, 1)
        for k in range(4):
            for b in range(4):
                w = F(0.5) * D[t][b] * S[z][k]
                w = fma(S[t][b], S[z][k], w)
                w = fma(F(0.5) * S[t][b], D[z][k], w)
                w = fma(third * D[t][b], D[z][k], w)
                acc = np.zeros_like(w)
                for a in range(3):
                    acc = fma(cw * D[d][a], w, acc)
                    m = {d: a, t: b, z: k}
                    i = [base[e] + m[e] for e in range(3)]
                    v = fma(acc, q, F(12582912.0)).view(np.int32).astype(np.int64) - 0x4B400000
                    np.add.at(J[d], (i[2], i[1], i[0]), v)
    return J.astype(np.int32).astype(F) * (F(items) * wmax * F(1.0 / 536870912.0))


def electrons(lo, tile, dx, dt, n, rng):
    """Positions in a tile and momenta, with the cells and offsets that they are kept as."""
    X = rng.uniform(lo, [lo[d] + tile[d] for d in range(3)], (6 * n, 3))
    x, u = X * dx, momenta(6 * n, rng)
    cell = np.floor(x / dx)
    o = (x / dx - cell).astype(F)
    d0, v, dtdx = o - (o >= F(0.5)).astype(F), u * F(0.5), F(dt * (1.0 / dx))
    ok = ((o < 1) & (d0 + dtdx * v == fma(np.full_like(v, dtdx), v, d0))).all(1)
    assert ok.sum() >= n
    return x[ok][:n], u[ok][:n], cell[ok][:n].astype(int), o[ok][:n]


@pytest.mark.parametrize("tile", [(16, 8, 4), (8, 8, 8), (12, 5, 6)])      # pitches 24 x 13, 16 x 13 and general
def test_current_bit_for_bit(P, tile):
    n, items = (48, 40, 40), 600
    lo = tuple(tile[d] * -(-16 // tile[d]) for d in range(3))
    w = small_3d().with_(n=n, beam=synth.BEAM_NONE, slab_lo=lo, slab_hi=tuple(lo[d] + tile[d] for d in range(3)))
    rng = np.random.default_rng(sum(tile))
    sim = P.Simulation(P.config_from(w, tile=tile, chunk=4096, max_particles=items))
    dx, dt = w.dx, sim.info().params.dt
    x, u, cell, o = electrons(lo, tile, dx, dt, items, rng)
    wt = (w.n_e * rng.uniform(0.5, 1.0, items)).astype(F)
    sim.set_particles(x, u.astype(np.float64), wt.astype(np.float64), np.arange(items))
    sim.step(1)
    p = sim.particles()
    np.testing.assert_array_equal(p["u"][np.argsort(p["id"])], u)          # no force: as given
    got = sim.fields()[6:]
    sim.close()
    np.testing.assert_array_equal(got.astype(F), current(cell, o, u, wt, n, dx, dt, items))
