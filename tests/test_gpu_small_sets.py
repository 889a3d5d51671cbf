"""Levels of many small sets: the tau kernel's shape is the tuner's choice there
too (the 256-wide tiles that the largest levels run without trials would be
nearly empty), and tuned and untuned runs take the same steps."""
import numpy as np
import pytest

from paper_1407_7105_gb300 import ics

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [5, 64])
def test_many_small_sets_are_tuned(cclib, size):
    nsys, dt = 4400, 1 / 256
    one = [ics.plummer(size, seed=s) for s in range(4)]
    m, x, v = (np.concatenate([one[k % 4][q] for k in range(nsys)], axis=-1) for q in range(3))
    out = []
    for autotune in (1, 0):
        c = cclib.Context(m, x, v, dt=dt, s_small=0, autotune=autotune)
        c.set_systems(np.arange(nsys + 1) * size)
        c.evolve(dt)
        pairs = nsys * size * (size - 1) // 2
        cells = [e for e in c.tuning() if e["kernel"] == "tau_mixed" and e["bin"] == pairs.bit_length() - 1]
        assert bool(cells) == bool(autotune)
        out.append(c.get_state()[2:])
        c.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
