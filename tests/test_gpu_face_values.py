"""A face value that the interface ignores (zero-flux and periodic faces) stays
ignored by every pass, also where a float cannot hold it: the fields are bitwise
those of the same grid with value 0."""
import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa
from helpers import make_grid, run_gpu
from paper_2209_13768_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, ZF, P = "dirichlet", "zeroflux", "periodic"
FACES = {
    "walls": [ZF] * 6,
    "x": [P, P, ZF, ZF, ZF, D],
    "yz": [ZF, ZF] + [P] * 4,
}


def _problem(shape, faces, value, kvar, steps=6):
    rng = np.random.default_rng(1)
    k = np.exp(0.5 * rng.standard_normal(shape[::-1])).astype(np.float32) if kvar else 0.8
    return W.Problem(shape=shape, T0=rng.uniform(0, 1, shape[::-1]).astype(np.float32), k=k, u=(0.0, 0.0, 0.0),
                     bc=[(kind, 0.5 if kind == D else value) for kind in FACES[faces]], steps=steps)


@pytest.mark.parametrize("value", [-7.5, 1e300])
@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("faces", sorted(FACES))
@pytest.mark.parametrize("shape", [(64, 5, 7), (120, 9, 5), (125, 12, 6)])
def test_ignored_face_values(shape, faces, kvar, storage, value):
    zero, p = (_problem(shape, faces, v, kvar) for v in (0.0, value))
    ref = run_gpu(zero, storage=storage, variant=-1)
    for variant in (-1, 3, 5, 7):
        np.testing.assert_array_equal(run_gpu(p, storage=storage, depth=2, variant=variant), ref, err_msg=f"variant {variant}")
    with make_grid(p, storage=storage) as g:
        wfa.batch_run([g], [p.steps])
        np.testing.assert_array_equal(g.read_field(), ref, err_msg="batch")
