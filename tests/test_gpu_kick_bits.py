"""The FP64 kick against the oracle bit for bit: both do the same operations in
the same order, whether a product or r^-3 is taken by the integer and FP32 pipes
(exponents within 2^+-200) or by the IEEE instructions, and whether the forces are
computed in place (below 2^21 pairs, 2048 bodies) or read from the matrices."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1407_7105_gb300 import ics

pytestmark = pytest.mark.gpu


def _bodies(n, seed, scale, masses):
    """Coordinates over six decades around `scale` (at 2^+-100 the squares, at
    2^+-200 the differences of one row lie on both sides of the range), some of
    them shared or zero; masses equal, over four decades, or over the range's edge."""
    rng = np.random.default_rng(seed)
    x = np.sign(rng.standard_normal((3, n))) * 10.0 ** rng.uniform(-3, 3, (3, n)) * scale
    k = n // 3
    x[0, :k] = x[0, 0]
    x[1, k // 2:k] = 0.0
    m = np.full(n, 1.0 / n)
    if masses == "spread":
        m = 10.0 ** rng.uniform(-4, 0, n) / n
    elif masses == "edge":
        m = m * 2.0 ** rng.choice([-210.0, -195.0, 0.0, 195.0], n)
    return m, np.ascontiguousarray(x), np.zeros((3, n))  # (at rest: the velocity is the whole sum)


@pytest.mark.parametrize("n", [2, 9, 33, 300, 725, 1025, 2048, 2049, 2061])
@pytest.mark.parametrize("scale,eps,masses", [
    (1.0, 0.0, "equal"), (1.0, 0.0, "spread"), (1.0, 0.01, "spread"), (1.0, 0.0, "edge"),
    (2.0 ** 100, 0.0, "spread"), (2.0 ** -100, 0.0, "equal"), (2.0 ** -100, 2.0 ** -99, "spread"),
    (2.0 ** 200, 0.0, "equal"), (2.0 ** -200, 0.0, "spread")])
def test_kick_bits(cclib, n, scale, eps, masses):
    m, x, v = _bodies(n, n, scale, masses)
    rng = np.random.default_rng(n + 1)
    lab = np.arange(n, dtype=np.int32)
    g = rng.permutation(n)[: n // 2]
    if g.size:
        lab[g] = g.min()
    h = 1 / 64
    c = cclib.Context(m, x, v, eps=eps)
    c.kick(lab, h)
    _, _, _, gv = c.get_state()
    c.close()
    s = O.State(m, x, v)
    O.kick(s, O.params(eps=eps), np.arange(n), lab, h)
    assert np.isfinite(s.v3).all() and np.any(s.v3 != 0.0)
    assert np.array_equal(gv, s.v3)


@pytest.mark.parametrize("n", [2048, 2049, 2061])
def test_ok_step_bits(cclib, n):
    """The OK split's outer kick leaves its fast pairs out of the same sums."""
    m, x, v = ics.plummer(n, seed=5)
    dt = 1 / 256
    c = cclib.Context(m, x, v, dt=dt, split=cclib.SPLIT_OK)
    c.evolve(dt)
    _, _, gx, gv = c.get_state()
    c.close()
    s = O.State(m, x, v)
    O.evolve(s, O.params(dt=dt, split=O.SPLIT_OK), 1)
    assert np.array_equal(gx, s.x3) and np.array_equal(gv, s.v3)
