"""Time-step graphs and components of cold states, where most relative speeds are
below what the tau kernel's common bounds certify and each pair's own separation
decides: the edges of the certified kernel are those of the FP64 tau of every pair
(near_tol above 1e-6 asks for that one), and the components those of the edges."""
import numpy as np
import pytest

from paper_1407_7105_gb300 import ics

pytestmark = pytest.mark.gpu


KINDS = ["cold", "rest", "some at rest", "masses", "stream", "collapse", "SI", "CGS"]


def _state(kind, n):
    m, x, v = ics.plummer(n, seed=9, Q=0.5, exact_scale=False)
    G = 1.0
    if kind == "cold":
        v = v * 1e-2
    elif kind == "rest":
        v = np.zeros_like(v)
    elif kind == "some at rest":
        v = v * np.where(np.arange(n) % 3 == 0, 0.0, 1e-3)
    elif kind == "masses":
        m, v = ics.salpeter_masses(n, 3, 9100), v * 3e-2
    elif kind == "stream":  # together at a hundred times their own speeds
        v = v * 1e-2 + np.array([[30.0], [-40.0], [10.0]])
    elif kind == "collapse":
        v = -1e-2 * x
    elif kind == "SI":  # parsecs, a thousand Suns
        G, m, x, v = 6.674e-11, m * 2e33, x * 3.1e16, v * 2.1
    elif kind == "CGS":
        G, m, x, v = 6.674e-8, m * 2e36, x * 3.1e18, v * 210.0
    return G, m, np.ascontiguousarray(x), np.ascontiguousarray(v)


# (components_noalloc takes 256-wide tiles from 3072 bodies, the graph from about 22000)
@pytest.mark.parametrize("n,kind", [(n, k) for n in (63, 257, 1000, 3100) for k in KINDS] + [(22100, "cold")])
def test_cold_graph(cclib, n, kind):
    import torch
    G, m, x, v = _state(kind, n)
    T = {"SI": 5e14, "CGS": 5e14}.get(kind, 1.0)  # an N-body time, roughly
    edged = 0
    for h in (T / 16, T / 256, T / 4096)[n > 20000:]:
        out = []
        for tol in (1e-12, 1e-5):
            c = cclib.Context(m, x, v, dt=T, eta=0.03, G=G, near_tol=tol)
            e, ne, _ = c.timestep_graph(h)
            lab, k = c.components(h)
            out.append((e, ne, lab, k))
            c.close()
        assert out[0][1] == out[1][1] and np.array_equal(out[0][0], out[1][0])
        edged += 0 < ne < n * (n - 1) // 2
        want = np.arange(n)
        while True:
            low = np.minimum(want[e[:, 0]], want[e[:, 1]])
            new = want.copy()
            np.minimum.at(new, e[:, 0], low)
            np.minimum.at(new, e[:, 1], low)
            new = new[new]
            if np.array_equal(new, want):
                break
            want = new
        dm, dx, dv = (torch.tensor(a, device="cuda") for a in (m, x, v))
        raw = torch.zeros(n, dtype=torch.int32, device="cuda")
        num = torch.zeros(1, dtype=torch.int64, device="cuda")
        cclib.components_noalloc(dm, dx, dv, h, raw, num, params=cclib.default_params(eta=0.03, G=G))
        for got, k in ((out[0][2], out[0][3]), (out[1][2], out[1][3]), (raw.cpu().numpy(), int(num.item()))):
            assert np.array_equal(got, want)
            assert k == np.count_nonzero(np.bincount(want) > 1)
    assert edged  # (a threshold with some edges and not all)
