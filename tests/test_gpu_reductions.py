"""The field sum and the stability limit at the sizes where their row kernels
can go wrong: rows around a thread's 4 cells and a warp's 128, every face
kind, values whose fp32 sums leave the range, tiny next to large.

Tolerances. The sum adds 4 cells exactly (fp32 with its error terms) and the
rest in fp64: a few thousand additions a thread and 2^10 partials keep it
within 1e-13 of sum |T|. The limit is the fp64 maximum over the cells, the
oracle's expression term for term: 1e-14.
"""
import numpy as np
import pytest

import oracle
import paper_2209_13768_gb300 as wfa
from paper_2209_13768_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, ZF, P, DC = W.D, W.ZF, W.P, W.DC
SHAPES = [(2, 2, 2), (3, 3, 5), (4, 9, 3), (31, 6, 4), (127, 5, 3), (128, 4, 4), (129, 3, 7), (130, 33, 40), (514, 3, 3)]


@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
@pytest.mark.parametrize("shape", SHAPES)
def test_total_heat_is_the_fp64_sum(shape, storage):
    rng = np.random.default_rng(sum(shape))
    for scale in ("unit", "mixed", "huge"):
        T = rng.uniform(-1, 1, shape[::-1])
        if scale == "mixed":
            T = T * np.exp2(rng.integers(-40, 40, T.shape))
        if scale == "huge":   # four of them overflow fp32
            T = np.where(rng.random(T.shape) < 0.5, 3.0e38, 1.0)
        with wfa.Grid(shape, storage=storage) as g:
            g.set_field(T.astype(np.float32))
            held = g.read_field().astype(np.float64)
            got = g.total_heat()
        assert abs(got - held.sum()) <= 1e-13 * np.abs(held).sum(), scale


def test_total_heat_of_infinities():
    T = np.ones((3, 4, 9), np.float32)
    T[1, 2, 3] = np.inf
    with wfa.Grid((9, 4, 3)) as g:
        g.set_field(T)
        assert g.total_heat() == np.inf
        T[1, 2, 5] = -np.inf
        g.set_field(T)
        assert np.isnan(g.total_heat())


@pytest.mark.parametrize("faces", [[(D, 0.0)] * 6, [(ZF, 0)] * 6, [(P, 0)] * 6,
                                   [(P, 0), (P, 0), (D, 0.0), (ZF, 0), (DC, 1.0), (D, 0.0)],
                                   [(DC, 1.0), (ZF, 0), (P, 0), (P, 0), (P, 0), (P, 0)]])
@pytest.mark.parametrize("shape", SHAPES[1:])   # held layers need an edge of 3
def test_stability_limit_by_rows(shape, faces):
    rng = np.random.default_rng(shape[0])
    for spread in (0.5, 3.0):
        k = np.exp(spread * rng.standard_normal(shape[::-1])).astype(np.float32)
        for at in (None, 0, shape[0] // 2, shape[0] - 1):   # the largest values at an x face or inside
            kk = k.copy()
            if at is not None:
                kk[-1, -1, at] = kk[0, 0, at] = 40.0 * k.max()
            with wfa.Grid(shape, h=(1.0, 0.8, 1.1)) as g:
                g.set_bcs(faces)
                g.set_coeffs(kk)
                got = g.stability_dt()
            ref = oracle.dt_max(shape=shape, h=(1.0, 0.8, 1.1), k=kk.astype(np.float64), bc=faces)
            assert got == pytest.approx(ref, rel=1e-14)
