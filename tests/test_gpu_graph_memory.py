"""The time-step graph of a dense state holds no more device memory when its edges
come from the certified kernel's records than when the FP64 kernels write them
(near_tol above 1e-6), but for the records that a level keeps anyway; and a list
longer than those is complete."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _held(cclib, ic, **kw):
    import torch
    c = cclib.Context(*ic, **kw)
    c.timestep_graph(1e-9)  # (the level's own buffers)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    E, ne, _ = c.timestep_graph(1e6)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    c.close()
    return held, E, ne


@pytest.mark.parametrize("edge_rec_max", [0, 100])
def test_dense_graph(cclib, plummer_ic, edge_rec_max):
    n = 6000
    ic = plummer_ic(n, seed=9)
    plain, _, _ = _held(cclib, ic, near_tol=1e-3)
    held, E, ne = _held(cclib, ic, edge_rec_max=edge_rec_max)
    i, j = np.triu_indices(n, 1)
    assert ne == i.size and np.array_equal(E, np.stack([i, j], axis=1))
    assert held <= plain + (1 << 24), (held / ne, plain / ne)
