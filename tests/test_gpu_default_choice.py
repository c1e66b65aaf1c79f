"""The untuned choice between one and two steps a pass, on both sides of its
lines: tiles that n_x or n_y fill well or badly, few planes, ragged periodic
rows. Whatever is chosen gives bitwise the plain one-column kernel's field."""
import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa

pytestmark = pytest.mark.gpu

D, ZF, P = "dirichlet", "zeroflux", "periodic"
FACES = {"cold": [(D, 0.5)] * 6, "channel": [(P, 0.0)] * 2 + [(ZF, 0.0)] * 4, "torus": [(P, 0.0)] * 6}


@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
@pytest.mark.parametrize("shape,faces,kvar,depth", [
    ((128, 128, 128), "cold", True, 2), ((200, 97, 51), "cold", True, 2), ((250, 97, 41), "cold", True, 1),
    ((1000, 1000, 2), "cold", True, 1), ((700, 2, 700), "cold", True, 1),
    ((200, 160, 137), "torus", True, 2), ((57, 160, 482), "torus", True, 1), ((25, 160, 1100), "channel", True, 2),
    ((480, 160, 57), "torus", False, 2), ((481, 160, 57), "torus", False, 1), ((481, 160, 57), "channel", False, 1),
    ((176, 81, 300), "torus", False, 1), ((1050, 4, 1001), "torus", False, 1), ((200, 160, 137), "channel", False, 2),
    ((124, 131, 126), "cold", False, 2), ((121, 131, 126), "cold", False, 1),
])
def test_default_choice(shape, faces, kvar, depth, storage):
    rng = np.random.default_rng(shape[0])
    T = rng.random(shape[::-1], dtype=np.float32)
    out = []
    for variant in (0, -1):
        with wfa.Grid(shape, storage=storage) as g:
            g.set_bcs(FACES[faces])
            g.set_coeffs(T + 0.5 if kvar else 0.7)
            g.set_field(T)
            g.set_dt(0.05)
            g.set_tuning(0, variant)
            if variant == 0:
                assert g.tuning()[0] == depth
            for n in (2, 3):
                g.step(n)
            out.append(g.read_field())
    np.testing.assert_array_equal(*out)
