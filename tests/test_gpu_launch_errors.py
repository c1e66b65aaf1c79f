"""A launch that the device refuses is reported by the call that made it, and
by no other."""
import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [3, 5, 7])
def test_refused_launch_is_reported_once(variant):
    shape = (8, 2, 65536)   # one plane a chunk: one block more along z than a launch may have
    T = np.ones(shape[::-1], np.float32)
    with wfa.Grid(shape) as g, wfa.Grid((8, 4, 4)) as other:
        for x in (g, other):
            x.set_coeffs(1.0)
            x.set_dt(0.1)
        g.set_field(T)
        g.set_tuning(1, variant)
        g.set_zchunk(1)
        with pytest.raises(wfa.WfaError):
            g.step(1 if variant != 7 else 2)
        other.set_field(np.ones((4, 4, 8), np.float32))
        other.step(3)
        np.testing.assert_array_equal(other.read_field(), 1.0)
        g.set_zchunk(0)
        g.step(2)
        np.testing.assert_array_equal(g.read_field(), T)
