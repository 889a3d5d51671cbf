"""The tau kernel's bounds for single pairs (tau_pair_bounds and the sums the
kernel takes signs of, csrc/cc_device.cuh / cc_mixed.cu), restated in numpy
float32 and checked against the oracle's FP64 tau: no pair they certify has
tau < h.  Differences are formed from the rounded high parts, as the kernel
forms them, with the raised r_min and v_thr of the rows' largest |x|, |v|."""
import numpy as np
import pytest

from oracle import oracle as O

f32 = np.float32
U32 = f32(2.0 ** -24)


def constants(eta, h, outside):
    """mixed_tau_params"""
    eta_in = 1.0 if outside else eta
    etah = eta_in * eta / h if outside else eta / h
    hq = h / eta if outside else h
    M, D = 1.02, max(1.0 / 32, 0.75 * eta_in / (2.0 + eta_in))
    c = M * (2.0 + eta_in) / (2.0 * etah * (1.0 - D))
    q = hq / c
    if not 0.75 * M * q < 0.95:
        return None
    T = M / (etah * (1.0 - 0.75 * M * q))
    return f32(c * c * 1.0001), f32(T * T * 1.0001), f32(M * eta_in / (2.0 * etah * D) * 1.0001)


def certified(dx, dv, mu, amax, vabs, k, eps2=0.0):
    """tau_pair_bounds and the kernel's two sums, float32 step by step"""
    c2, t2, v = k
    mu = f32(mu) * f32(1.0001)
    r3 = mu * t2
    rmin = f32(1.0005) * f32(np.exp2(np.log2(r3) / f32(3)))
    rmin = max(rmin, f32(1.02e3) * f32(7.1) * U32 * f32(amax), f32(1e-15))
    vt = max(f32(1.0001) * v * mu / (rmin * rmin), f32(1.02e3) * f32(7.1) * U32 * f32(vabs), f32(1e-15))
    w2 = vt * vt
    p2 = max(rmin * rmin, f32(1.0001) * c2 * w2)
    if not (1e-36 < r3 < 1e36 and w2 < 1e30 and p2 < 1e30):
        return np.zeros(dx.shape[1], dtype=bool)
    p, w = f32(eps2) - p2, -w2
    for q in range(3):
        p = (dx[q] * dx[q] + p).astype(f32)
        w = (dv[q] * dv[q] + w).astype(f32)
    return (w >= 0) & ((p - c2 * w).astype(f32) >= 0)


def pairs(rng, n, X, V):
    """bodies around points up to X from the origin, separations and speeds
    over many scales; a third approach head on, a third slowly"""
    xi, vi = rng.uniform(-X, X, (3, n)), rng.uniform(-V, V, (3, n))
    dx = rng.standard_normal((3, n)) * np.exp(rng.uniform(-7, 2, n))
    dv = rng.standard_normal((3, n)) * np.exp(rng.uniform(-6, 1, n))
    head = dx / np.linalg.norm(dx, axis=0)
    dv[:, ::3] = -head[:, ::3] * np.linalg.norm(dv[:, ::3], axis=0)
    dv[:, 1::3] = -head[:, 1::3] * np.exp(rng.uniform(-12, -2, dv[:, 1::3].shape[1]))
    return xi, xi + dx, vi, vi + dv


@pytest.mark.parametrize("outside", [0, 1])
@pytest.mark.parametrize("eta", [0.0025, 0.03, 0.4, 1.5])
@pytest.mark.parametrize("X,V", [(1.0, 1.0), (300.0, 30.0)])
@pytest.mark.parametrize("eps", [0.0, 1 / 256])
def test_certified_pairs_are_no_edges(outside, eta, X, V, eps):
    rng = np.random.default_rng(int(1e4 * eta) + outside)
    n = 3000
    xi, xj, vi, vj = pairs(rng, n, X, V)
    mi, mj = 2e-4, 1e-4
    p = O.params(eta=eta, eps=eps, eta_outside=bool(outside))
    tau = np.array([O.tau_parts(xi[:, k], vi[:, k], mi, xj[:, k], vj[:, k], mj, p)[0] for k in range(n)])
    dx, dv = xj.astype(f32) - xi.astype(f32), vj.astype(f32) - vi.astype(f32)
    some = 0
    for h in (2.0 ** -10, 2.0 ** -8, 2.0 ** -6, 0.25):
        k = constants(eta, h, outside)
        if k is None:
            continue
        ok = certified(dx, dv, mi + mj, X, V, k, eps * eps)
        some += int(ok.sum())
        assert np.all(tau[ok] >= h), (h, tau[ok].min())
    if X == 1.0 and eta == 0.03 and not outside:
        assert some > n // 2  # the bounds settle a good share
    # each pair's own tau, barely an edge: no bound may certify it
    for j in range(0, n, 11):
        for rel in (0.999, 0.99):
            k = constants(eta, float(tau[j]) / rel, outside) if np.isfinite(tau[j]) and tau[j] > 0 else None
            if k is not None:
                assert not certified(dx[:, j:j + 1], dv[:, j:j + 1], mi + mj, X, V, k, eps * eps)[0], (j, tau[j])


def test_a_looser_bound_is_seen():
    """with the free-fall bound dropped (r_min at its floor) the test fails"""
    rng = np.random.default_rng(3)
    xi, xj, vi, vj = pairs(rng, 3000, 1.0, 1.0)
    p = O.params(eta=0.03)
    tau = np.array([O.tau_parts(xi[:, k], vi[:, k], 1e-2, xj[:, k], vj[:, k], 1e-2, p)[0] for k in range(3000)])
    c2, t2, v = constants(0.03, 2.0 ** -6, 0)
    bad = certified(xj.astype(f32) - xi.astype(f32), vj.astype(f32) - vi.astype(f32), 2e-2, 1e-6, 1e-6,
                    (c2, f32(1e-30), f32(1e-30)))
    assert (tau[bad] < 2.0 ** -6).any()
