"""cc_timestep_graph and cc_components_noalloc on the certified tau kernel:
edge lists and labels equal to the oracle's FP64 ones at the edges of the
kernel's tiles and column chunks, for cold states (nearly every pair below
the certificates' speed bound), states whose coordinates lie outside the
certificates' range, and unequal masses; and the graph's two ways (certified,
and FP64 for a near_tol the FP32 bounds cannot see) against each other."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1407_7105_gb300 import ics

pytestmark = pytest.mark.gpu


def _noalloc(cclib, m, x, v, h, **kw):
    import torch
    d = [torch.tensor(a, device="cuda") for a in (m, x, v)]
    lab = torch.full((m.shape[0],), -5, dtype=torch.int32, device="cuda")
    k = torch.full((1,), -5, dtype=torch.int64, device="cuda")
    cclib.components_noalloc(*d, h, lab, k, params=cclib.default_params(**kw))
    return lab.cpu().numpy(), int(k.item())


def _check(cclib, m, x, v, h, eps=0.0):
    s, p = O.State(m, x, v), O.params(eps=eps)
    oE, onear = O.edges(s, p, h)
    olab, ok = O.components(s, p, h)
    c = cclib.Context(m, x, v, eps=eps)
    E, ne, near = c.timestep_graph(h)
    c.close()
    assert ne == oE.shape[0] and near == onear and np.array_equal(E, oE)
    w = cclib.Context(m, x, v, eps=eps, near_tol=1e-3)  # the FP64 tau of every pair
    Ew, new, nearw = w.timestep_graph(h)
    w.close()
    assert new == ne and np.array_equal(Ew, oE) and nearw >= near
    lab, k = _noalloc(cclib, m, x, v, h, eps=eps)
    assert k == ok and np.array_equal(lab, olab)
    return ne


@pytest.mark.parametrize("n", [2, 31, 33, 63, 64, 65, 97, 127, 128, 129, 255, 256, 257, 513, 1031, 6143, 6151])
def test_tile_edges(cclib, plummer_ic, n):
    m, x, v = plummer_ic(n, seed=3)
    ne = _check(cclib, m, x, v, 1 / 100)
    assert n < 100 or ne > 0


@pytest.mark.parametrize("kind", ["cold", "still", "far", "huge", "masses", "soft"])
def test_states_the_bounds_do_not_fit(cclib, plummer_ic, kind):
    n, h, eps = 700, 1 / 64, 0.0
    m, x, v = plummer_ic(n, seed=5)
    rng = np.random.default_rng(1)
    if kind == "cold":
        v = v * 1e-3
    elif kind == "still":
        v = np.zeros_like(v)
    elif kind == "far":
        x = x + 1e6
    elif kind == "huge":  # coordinates beyond 1e15: T_ff scales with r^1.5, T_fb with r
        x, v, h = x * 1e16, v * 1e-8, h * 1e24
    elif kind == "masses":
        m = m * np.exp(rng.uniform(-8, 8, n))
    else:
        eps = 0.05
    _check(cclib, np.ascontiguousarray(m), np.ascontiguousarray(x), np.ascontiguousarray(v), h, eps)


@pytest.mark.parametrize("what,bad", [("v", np.inf), ("v", np.nan), ("x", np.nan), ("m", np.nan), ("m", 0.0)])
def test_noalloc_on_values_no_context_takes(cclib, plummer_ic, what, bad):
    """cc_components_noalloc does not look at the values: a body with one that
    cc_init refuses gets the FP64 predicate's answer, pair by pair."""
    n, h, at = 300, 1 / 100, 77
    m, x, v = (np.array(a) for a in plummer_ic(n, seed=6))
    (m if what == "m" else x[1] if what == "x" else v[2])[at] = bad
    lab, k = _noalloc(cclib, m, x, v, h)
    s, p = O.State(m, x, v), O.params()
    i, j = np.triu_indices(n, 1)
    with np.errstate(all="ignore"):
        on = np.array([O.tau_ids(s, p, int(a), int(b)) < h for a, b in zip(i, j)])
    want = np.arange(n)
    while True:
        low = np.minimum(want[i[on]], want[j[on]])
        new = want.copy()
        np.minimum.at(new, i[on], low)
        np.minimum.at(new, j[on], low)
        if np.array_equal(new, want):
            break
        want = new
    assert np.array_equal(lab, want)
    assert k == int((np.bincount(want) >= 2).sum())


@pytest.mark.parametrize("n", [2, 46, 64, 511, 512, 513, 600])
def test_graph_of_every_pair_is_sorted(cclib, n):
    """Every pair an edge: the edge list in order, at sizes around the sort's
    tiles (1024 keys: 46 bodies have 1035 pairs) and around the 128 tiles up to
    which the scatter scans the histograms itself (512: 130816 pairs, 513:
    131328)."""
    m, x, v = ics.plummer(n, seed=n, exact_scale=False)
    c = cclib.Context(m, x, v)
    edges, count, _ = c.timestep_graph(1e4, cap=n * n)
    c.close()
    i, j = np.triu_indices(n, 1)
    assert count == i.size
    assert np.array_equal(edges, np.stack([i, j], axis=1))
