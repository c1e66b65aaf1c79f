"""The row kernels of classic CG (cg_dir, cg_res) where they can go wrong: the
x extent around a thread's 4 cells and around the 8 / 16-lane tiles, odd and
single rows at the block's edge, z extents around the chunks, grids on both
sides of the block count up to which cg_res sums p.q itself, and breakdowns.

Tolerance. rtol = 0 runs exactly m iterations on both sides, so the iterates
are compared with the FP64 oracle's: fp32 rounding of each product amplified
by no more than the condition number of A (at most about 40 here) stays below
1e-5 relative to max |T|, as for the other fixed-iteration comparisons.
"""
import os

import numpy as np
import pytest

import oracle
import paper_2209_13768_gb300 as wfa
from paper_2209_13768_gb300 import workloads as W
from helpers import rel_linf

pytestmark = pytest.mark.gpu

D, ZF, P, DC = W.D, W.ZF, W.P, W.DC
FACES = [
    [(D, 0.3), (ZF, 0), (DC, 1.0), (D, 0.0), (ZF, 0), (DC, 2.0)],
    [(DC, 0.25), (D, 0.75), (P, 0), (P, 0), (D, 0.1), (ZF, 0)],
    [(P, 0), (P, 0), (ZF, 0), (DC, 0.4), (P, 0), (P, 0)],
]
SHAPES = [(31, 31, 4), (32, 33, 5), (33, 16, 17), (34, 15, 6), (63, 17, 3), (64, 32, 33), (65, 3, 16), (67, 18, 31),
          (129, 5, 47)]


def _problem(faces, shape, kvar, seed):
    rng = np.random.default_rng(seed)
    nx, ny, nz = shape
    k = np.exp(0.5 * rng.standard_normal((nz, ny, nx))).astype(np.float32) if kvar else 0.8
    T0 = rng.uniform(0, 1, (nz, ny, nx)).astype(np.float32)
    return W.Problem(shape=shape, T0=T0, k=k, bc=FACES[faces], h=(1.0, 0.9, 1.1))


def _run(p, dt, m, loop=None):
    if loop:
        os.environ["WFA_CG_LOOP"] = loop
    try:
        with wfa.Grid(p.shape, h=p.h) as g:
            g.set_bcs(p.bc)
            g.set_coeffs(p.k)
            g.set_field(p.T0)
            it, _ = g.implicit_step(dt, 1, rtol=0.0, max_iter=m)
            return it, g.read_field()
    finally:
        os.environ.pop("WFA_CG_LOOP", None)


def _check(p, m=6):
    k = p.k if np.isscalar(p.k) else np.asarray(p.k, dtype=np.float64)
    dt = 3.0 * oracle.dt_max(shape=p.shape, h=p.h, k=k, bc=p.bc)
    ref, it_ref, _ = oracle.implicit(p.T0, 1, shape=p.shape, h=p.h, k=k, bc=p.bc, dt=dt, rtol=0.0, max_iter=m)
    it, T = _run(p, dt, m)
    assert it == it_ref == m
    assert rel_linf(T, ref) <= 1e-5
    it_h, T_h = _run(p, dt, m, loop="host")
    assert it_h == it
    np.testing.assert_array_equal(T, T_h)


@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("faces", range(len(FACES)))
@pytest.mark.parametrize("shape", SHAPES)
def test_iterates_match_oracle_at_tile_edges(shape, faces, kvar):
    _check(_problem(faces, shape, kvar, seed=sum(shape) + faces))


@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("shape", [(130, 100, 40), (210, 161, 66)])   # p.q summed by cg_res; by cg_dir's last block
def test_iterates_match_oracle_larger(shape, kvar):
    _check(_problem(0, shape, kvar, seed=7))


def test_exact_solution_breaks_down_cleanly():
    # T constant on zero-flux faces solves the step: r = 0, so with rtol = 0
    # the first p.q is 0 and the solve ends with the field as it was
    shape = (66, 19, 9)
    p = W.Problem(shape=shape, T0=np.full(shape[::-1], 0.5, np.float32), k=0.8, bc=[(ZF, 0)] * 6, h=(1.0, 1.0, 1.0))
    it, T = _run(p, 1.0, 50)
    assert it <= 1
    np.testing.assert_array_equal(T, p.T0)
