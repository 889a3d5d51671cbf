"""cc_components_noalloc takes the masses as they are: with negative ones among
them (a pair's G (m_i + m_j) can cancel, or be negative) the labels are still
those of the FP64 predicate, pair by pair."""
import numpy as np
import pytest

from oracle import oracle as O

pytestmark = pytest.mark.gpu


def _labels(cclib, m, x, v, h):
    import torch
    d = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in (m, x, v)]
    lab = torch.full((m.shape[0],), -5, dtype=torch.int32, device="cuda")
    k = torch.full((1,), -5, dtype=torch.int64, device="cuda")
    cclib.components_noalloc(*d, h, lab, k)
    return lab.cpu().numpy()


def _want(m, x, v, h):
    n = m.shape[0]
    s, p = O.State(m, x, v), O.params()
    i, j = np.triu_indices(n, 1)
    on = np.array([O.tau_ids(s, p, int(a), int(b)) < h for a, b in zip(i, j)])
    want = np.arange(n)
    while True:
        low = np.minimum(want[i[on]], want[j[on]])
        new = want.copy()
        np.minimum.at(new, i[on], low)
        np.minimum.at(new, j[on], low)
        if np.array_equal(new, want):
            return want
        want = new


@pytest.mark.parametrize("part", [1.25e-7, 1e-7, 3.3e-9, -1e-7])
@pytest.mark.parametrize("rel", [0.9, 0.99, 1.01, 1.1])
def test_masses_that_cancel(cclib, part, rel):
    m, x, v = np.array([1.0, -(1.0 - part)]), np.zeros((3, 2)), np.zeros((3, 2))
    x[0, 1] = 1e-3
    h = rel * 0.03 * np.sqrt(1e-9 / abs(part))
    assert np.array_equal(_labels(cclib, m, x, v, h), _want(m, x, v, h))


@pytest.mark.parametrize("slow", [1.0, 0.1, 1e-3])
@pytest.mark.parametrize("heavy", [1.0, 300.0])
def test_signs_mixed(cclib, plummer_ic, slow, heavy):
    n = 200
    m, x, v = plummer_ic(n, seed=8)
    m = m * np.where(np.arange(n) % 3 == 1, -heavy, 1.0)
    for h in (1 / 8, 1 / 32):
        assert np.array_equal(_labels(cclib, m, x, v * slow, h), _want(m, x, v * slow, h)), h
