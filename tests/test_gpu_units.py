"""States in other units than N-body ones, where products of the FP32 decision
leave the floats' range (r mu in CGS or SI units, r^2 of tiny lengths): graph,
components and steps of every split equal to the oracle's FP64 ones."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1407_7105_gb300 import ics

pytestmark = pytest.mark.gpu

SUN, AU, PC = 1.989e30, 1.496e11, 3.0857e16
CGS, SI = 6.674e-8, 6.674e-11
# (G, length, mass) of a sphere of total mass 1 in N-body units
UNITS = {"cgs_au": (CGS, 1e2 * AU, 1e3 * SUN * 100), "cgs_pc": (CGS, 1e2 * PC, 1e3 * SUN * 1e4),
         "si_au": (SI, AU, SUN * 100), "si_3pc": (SI, 3 * PC, SUN * 1e4), "si_kpc": (SI, 1e3 * PC, SUN * 1e8),
         "tiny": (1.0, 1e-20, 1.0), "light": (1.0, 1.0, 1e-40), "large_G": (1e30, 1e10, 1e-20)}


def _sphere(n, unit, seed=3):
    G, L, M = UNITS[unit]
    m, x, v = ics.plummer(n, seed=seed)
    V = np.sqrt(G * M / L)
    return m * M, x * L, v * V, G, L / V


def _graph(cclib, m, x, v, h, G):
    import torch
    s, p = O.State(m, x, v), O.params(G=G)
    oE, _ = O.edges(s, p, h)
    olab, ok = O.components(s, p, h)
    c = cclib.Context(m, x, v, G=G)
    E, ne, _ = c.timestep_graph(h)
    lab, k = c.components(h)
    c.close()
    assert ne == oE.shape[0] and np.array_equal(E, oE)
    assert k == ok and np.array_equal(lab, olab)
    d = [torch.tensor(a, device="cuda") for a in (m, x, v)]
    lab = torch.full((m.shape[0],), -5, dtype=torch.int32, device="cuda")
    k = torch.full((1,), -5, dtype=torch.int64, device="cuda")
    cclib.components_noalloc(*d, h, lab, k, params=cclib.default_params(G=G))
    assert int(k.item()) == ok and np.array_equal(lab.cpu().numpy(), olab)
    return ne


def test_pairs_that_are_no_edges(cclib):
    """Two Suns an astronomical unit apart (CGS, h = 1 s), stars of 100 Suns 3 pc
    apart and a star 100 AU from 4e6 Suns (SI): tau is 290 h and more."""
    z = np.zeros((3, 2))
    for ma, mb, r, vel, h, G in ((1e3 * SUN, 1e3 * SUN, 1e2 * AU, 3e6, 1.0, CGS),
                                 (100 * SUN, 100 * SUN, 3 * PC, 600.0, 1e11, SI),
                                 (4e6 * SUN, SUN, 100 * AU, 6e6, 1.0, SI)):
        x, v = z.copy(), z.copy()
        x[0, 1], v[1, 1] = r, vel
        assert _graph(cclib, np.array([ma, mb]), x, v, h, G) == 0


@pytest.mark.parametrize("unit", sorted(UNITS))
@pytest.mark.parametrize("frac", [1 / 16, 1 / 100, 1 / 1000])
def test_graph_and_components(cclib, unit, frac):
    m, x, v, G, T = _sphere(400, unit)
    ne = _graph(cclib, m, x, v, T * frac, G)
    assert frac < 0.01 or ne > 0


@pytest.mark.parametrize("unit", sorted(UNITS))
@pytest.mark.parametrize("kind", ["cc0", "cc32", "cc512", "hold", "ok", "systems"])
def test_step(cclib, unit, kind):
    """One step of the FP64 form on the level kernels (s_small = 0), the warps' (32)
    and the batched kernel (512; many systems), bit for bit."""
    off = None
    if kind == "systems":
        G, L, M = UNITS[unit]
        m, x, v, off = ics.small_systems(24, seed=7, n_max=100)
        V = np.sqrt(G * M / L)
        m, x, v, T = m * M, x * L, v * V, L / V
    else:
        m, x, v, G, T = _sphere(400, unit)
    dt = T / 64
    kw = {"cc0": dict(s_small=0), "cc32": dict(s_small=32), "cc512": dict(s_small=512),
          "systems": dict(s_small=512), "hold": dict(split=cclib.SPLIT_HOLD), "ok": dict(split=cclib.SPLIT_OK)}[kind]
    c = cclib.Context(m, x, v, dt=dt, G=G, **kw)
    if off is not None:
        c.set_systems(off)
    c.evolve(dt)
    _, _, gx, gv = c.get_state()
    c.close()
    s = O.State(m, x, v)
    split = {"hold": O.SPLIT_HOLD, "ok": O.SPLIT_OK}.get(kind, O.SPLIT_CC)
    O.evolve(s, O.params(dt=dt, G=G, split=split), 1, sys_off=off)
    assert np.array_equal(gx, s.x3) and np.array_equal(gv, s.v3)
