"""The kick and the energy diagnostic at the sizes where their kernels change
shape: the FP64 kick below and above 2^18 pairs (in place, eight rows a block;
forces first, rows summed by warp pairs after), the mixed kick from 2^29 pairs
on (two columns at a time), the energy's triangle of tiles.

FP64 sums: a row of n - 1 terms has a rounding error of at most (n + 12) u
times the sum of the absolute terms (n - 1 additions; at most 13 roundings in a
term), here and in the oracle, so the two differ by at most twice that.  A pair
left out or taken twice shows up as ~1/n of that sum, 1e9 times as much."""
import numpy as np
import pytest

import _bounds as B
from oracle import oracle as O
from paper_1407_7105_gb300 import ics

pytestmark = pytest.mark.gpu


def _bodies(n, seed, scale=1.0):
    """Unequal masses over four decades, some coordinates shared (zero
    differences), the length unit times scale."""
    rng = np.random.default_rng(seed)
    m = 10.0 ** rng.uniform(-4, 0, n) / n
    x = rng.standard_normal((3, n))
    k = n // 3
    x[0, :k] = x[0, 0]
    x[1, k // 2:k] = x[1, k // 2]
    return m, np.ascontiguousarray(x * scale), np.zeros((3, n))


def _labels(n, seed):
    """Every body its own component, but for one large and some small ones."""
    rng = np.random.default_rng(seed)
    lab = np.arange(n, dtype=np.int32)
    g = rng.permutation(n)[: n // 2]
    lab[g[: n // 4]] = g[0] if g.size else 0
    for a in range(n // 4, g.size - 2, 3):
        lab[g[a:a + 3]] = g[a]
    return lab


# (724 bodies: 261726 pairs, 725: 262450, around 2^18 = 262144; 2^+-300: r^-3
# leaves the fast path's range of exponents)
@pytest.mark.parametrize("n", [2, 9, 31, 33, 129, 724, 725, 737, 1025])
@pytest.mark.parametrize("eps,scale", [(0.0, 1.0), (0.01, 1.0), (0.0, 2.0 ** 300), (0.0, 2.0 ** -300)])
def test_fp64_kick(cclib, n, eps, scale):
    m, x, v = _bodies(n, n, scale)
    lab = _labels(n, n + 1)
    h = 1 / 64
    c = cclib.Context(m, x, v, eps=eps)
    c.kick(lab, h)
    _, _, gx, gv = c.get_state()
    c.close()
    s = O.State(m, x, v)
    O.kick(s, O.params(eps=eps), np.arange(n), lab, h)
    assert np.array_equal(gx, x)
    S = B.abs_accel_sum(m, x, eps=eps, labels=lab)
    assert np.all(np.abs(gv - s.v3) <= 2 * (n + 12) * B.U64 * h * S + 2 * B.U64 * np.abs(s.v3))


# (32769 bodies: 536887296 pairs, the first level of 2^29; 32895 = 257 tiles less one)
@pytest.mark.parametrize("n,eps", [(32769, 0.0), (32895, 1 / 256)])
def test_packed_mixed_kick(cclib, n, eps):
    m, x, v = ics.plummer(n, seed=4, exact_scale=False)
    rng = np.random.default_rng(5)
    m = m * 10.0 ** rng.uniform(-2, 0, n)
    v = np.zeros_like(v)
    lab = np.arange(n, dtype=np.int32)
    lab[rng.choice(n, 601, replace=False)] = 7
    h = 1 / 256
    c = cclib.Context(m, x, v, eps=eps, precision=cclib.PREC_MIXED)
    c.kick(lab, h)
    _, _, _, gv = c.get_state()
    c.close()
    rows = np.unique(np.concatenate([np.array([0, 1, 7, 127, 128, n - 2, n - 1]),
                                     np.flatnonzero(lab == 7)[:20], rng.choice(n, 100, replace=False)]))
    d = x[:, None, :] - x[:, rows, None]
    r2 = (d * d).sum(axis=0) + eps * eps
    w = np.where(lab[rows][:, None] != lab[None, :], m / np.where(r2 > 0, r2, 1.0) ** 1.5, 0.0)
    ref = (w * d).sum(axis=2)
    S = B.abs_accel_sum(m, x, eps=eps, labels=lab, rows=rows)[rows]
    err = np.linalg.norm(gv[:, rows] / h - ref, axis=0)
    assert np.all(err <= B.K_MIXED * B.U32 * S), float((err / (B.K_MIXED * B.U32 * S)).max())


@pytest.mark.parametrize("sizes,eps", [([2], 0.0), ([3], 0.01), ([64], 0.0), ([65], 0.0), ([127], 0.01), ([128], 0.0),
                                       ([129], 0.0), ([255], 0.0), ([257], 0.01), ([1000], 0.0), ([4097], 0.0),
                                       ([1, 2, 127, 3, 129, 64], 0.0), ([300, 1, 1, 257], 0.01)])
def test_energy(cclib, sizes, eps):
    n = sum(sizes)
    m, x, _ = _bodies(n, n)
    x = x + 1e-3 * np.random.default_rng(2).standard_normal((3, n))
    v = np.random.default_rng(1).standard_normal((3, n))
    c = cclib.Context(m, x, v, eps=eps)
    off = np.concatenate([[0], np.cumsum(sizes)])
    if len(sizes) > 1:
        c.set_systems(off)
    E, P, L = c.energy()
    c.close()
    e, p, a, size = 0.0, np.zeros(3), np.zeros(3), 0.0
    for b0, b1 in zip(off[:-1], off[1:]):
        s = O.State(m[b0:b1].copy(), np.ascontiguousarray(x[:, b0:b1]), np.ascontiguousarray(v[:, b0:b1]))
        de, dp, da = O.energy(s, eps=eps)
        e, p, a = e + de, p + dp, a + da
        T = 0.5 * (m[b0:b1] * (v[:, b0:b1] ** 2).sum(axis=0)).sum()
        size += T + abs(de - T)
    # (n (n - 1) / 2 + n terms of one sign each in T and W)
    assert abs(E - e) <= 2 * (n * n / 2 + n + 12) * B.U64 * size
    assert np.all(np.abs(P - p) <= 2 * (n + 4) * B.U64 * (m * np.abs(v)).sum())
    assert np.all(np.abs(L - a) <= 2 * (n + 4) * B.U64 * 2 * (m * np.abs(x).max(axis=0) * np.abs(v).max(axis=0)).sum())


def test_packed_mixed_kick_with_com(cclib):
    """The same with far components taken through their centres of mass,
    against the FP64 form (per-body bound as elsewhere, 400 sampled bodies)."""
    m, x, v = ics.box_fractal(32771, seed=3)
    dt = 1 / 256
    out = []
    for prec in (cclib.PREC_FP64, cclib.PREC_MIXED):
        c = cclib.Context(m, x, v, dt=dt, theta=0.5, precision=prec, near_tol=1e-6)
        c.evolve(dt)
        _, _, _, gv = c.get_state()
        g = c.stats()
        out.append((gv, g, c.near_pairs(1 << 20)[0]))
        c.close()
    assert out[1][1]["com_pairs"] > 0
    rows = np.random.default_rng(1).choice(m.shape[0], 400, replace=False)
    rows = np.setdiff1d(rows, np.concatenate([B.near_bodies(out[0][2]), B.near_bodies(out[1][2])]))
    S = B.abs_accel_sum(m, x, rows=rows)
    w, _ = B.check_velocity_bound(out[1][0][:, rows], out[0][0][:, rows], S[rows], dt, out[0][1]["max_depth_seen"])
    print("packed, COM: max error / bound", w)
