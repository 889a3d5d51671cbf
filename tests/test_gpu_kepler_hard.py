"""Kepler pairs that start next to a tight pericentre, where the universal
equation's iteration creeps back from a far start or runs round a cycle of doubles:
every one is solved, and where the oracle (the classical equation) puts it.

Both compute from the same rounded state, so they differ by how it determines the
orbit: 1/a = 2/r - v^2/mu loses the factor 2a/r (r the separation that the step
starts from) of its 2^-53; the state in the middle of the step is rounded to 2^-53
of a and not of its r, which is another factor 2a/r there.  That moves the phase by
as much of a period or of the time, and a phase error dt moves the body by |v| dt.
Each half and each side has some ten roundings of that size, and r is known to as much there; 1024 allows for it."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


def hard_pairs(n, seed, M=1.0):
    rng = np.random.default_rng(seed)
    a = np.exp(rng.uniform(np.log(0.5), np.log(2.0), n))
    e = 1.0 - 10.0 ** rng.uniform(-6, -1, n)
    E = np.where(rng.random(n) < 0.5, -1, 1) * 10.0 ** rng.uniform(-4, 0.4, n)
    q = rng.uniform(0.1, 1.0, n)
    b = a * np.sqrt(1 - e * e)
    r = a * (1 - e * np.cos(E))
    w = np.sqrt(M / a ** 3)
    th = rng.uniform(0, 2 * np.pi, n)
    c, s = np.cos(th), np.sin(th)
    x, y = a * (np.cos(E) - e), b * np.sin(E)
    u, v = -a * a * w * np.sin(E) / r, a * b * w * np.cos(E) / r
    pos = np.array([c * x - s * y, s * x + c * y, np.zeros(n)])
    vel = np.array([c * u - s * v, s * u + c * v, np.zeros(n)])
    m = np.empty(2 * n)
    m[0::2], m[1::2] = M / (1 + q), M * q / (1 + q)
    x3, v3 = np.empty((3, 2 * n)), np.empty((3, 2 * n))
    for out, d in ((x3, pos), (v3, vel)):
        out[:, 0::2], out[:, 1::2] = d * m[1::2] / M, -d * m[0::2] / M
    return m, x3, v3, a, e, E


def separation(a, e, E0, t, M=1.0):
    """of the pair a time t later"""
    w = np.sqrt(M / a ** 3)
    ma = np.remainder(E0 - e * np.sin(E0) + w * t, 2 * np.pi)
    lo, hi = np.zeros_like(a), np.full_like(a, 2 * np.pi)
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        low = mid - e * np.sin(mid) < ma
        lo, hi = np.where(low, mid, lo), np.where(low, hi, mid)
    return a * (1 - e * np.cos(lo))


def bounds(a, e, E0, dt, M=1.0):
    P = 2 * np.pi * np.sqrt(a ** 3 / M)
    r0, rm, r1 = (separation(a, e, E0, t) for t in (0.0, 0.5 * dt, dt))
    k = 1024 * 2.0 ** -53 * (2 * a / r0 + (2 * a / rm) ** 2)
    v1 = np.sqrt(M * (2 / r1 - 1 / a))
    return k * (2 * a + v1 * (P + dt)), k * (v1 + M / r1 ** 2 * (P + dt))


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_hard_pairs(cclib, seed):
    n, dt = 20000, 8.0
    m, x, v, a, e, E = hard_pairs(n, seed)
    off = 2 * np.arange(n + 1)
    c = cclib.Context(m, x, v, dt=dt, eta=0.03, kepler=1)
    c.set_systems(off)
    c.evolve(dt)
    _, _, gx, gv = c.get_state()
    c.close()
    s = O.State(m, x, v)
    st = O.evolve(s, O.params(dt=dt, eta=0.03, kepler=1), 1, sys_off=off)
    assert st.kepler_calls == 2 * n
    bx, bv = bounds(a, e, E, dt)
    for got, want, b in ((gx, s.x3, bx), (gv, s.v3, bv)):
        d = got - want
        rel = np.linalg.norm(d[:, 0::2] - d[:, 1::2], axis=0)
        assert np.all(rel <= b), (float((rel / b).max()), int((rel > b).sum()))
