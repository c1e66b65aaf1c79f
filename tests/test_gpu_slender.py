"""Slender grids, on both sides of the sizes where a two-step pass would need
more blocks along y or z than a launch may have (65535): they run, and give
bitwise the field of the one-step column march."""
import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa

pytestmark = pytest.mark.gpu

D, ZF = "dirichlet", "zeroflux"
BC = [(D, 0.5), (D, 0.0), (ZF, 0.0), (ZF, 0.0), (D, 1.0), (ZF, 0.0)]


def _run(shape, storage, kvar, tuning, tune=False):
    n = shape[0] * shape[1] * shape[2]
    T = (np.arange(n, dtype=np.uint32) * np.uint32(2654435761) >> np.uint32(24)).astype(np.float32).reshape(shape[::-1])
    with wfa.Grid(shape, storage=storage) as g:
        g.set_bcs(BC)
        g.set_coeffs(0.5 + T / 256 if kvar else 0.7)
        g.set_field(T)
        g.set_dt(0.05)
        g.set_tuning(*tuning)
        if tune:
            g.autotune()
        g.step(3)
        return g.read_field()


# rows of blocks: sweep_pair 8 rows (fp32) or 4 (bf16), sweep_pair_k 10, 22 or 46; z chunks of 16 planes at least
@pytest.mark.parametrize("shape,storage,kvar", [
    ((40, 262140, 2), wfa.BF16, False), ((40, 262141, 2), wfa.BF16, False),
    ((40, 524280, 2), wfa.F32, False), ((40, 524281, 2), wfa.F32, False),
    ((65, 655352, 2), wfa.BF16, True), ((65, 655353, 2), wfa.BF16, True),
    ((40, 2, 1048561), wfa.F32, False), ((9, 3, 262145), wfa.F32, True),
])
def test_slender_grids_run(shape, storage, kvar):
    ref = _run(shape, storage, kvar, (1, 3))
    np.testing.assert_array_equal(_run(shape, storage, kvar, (0, 0)), ref)
    np.testing.assert_array_equal(_run(shape, storage, kvar, (2, 7)), ref)


def test_autotune_of_a_slender_grid():
    shape = (40, 262141, 2)
    np.testing.assert_array_equal(_run(shape, wfa.BF16, False, (0, 0), tune=True), _run(shape, wfa.BF16, False, (1, 3)))
