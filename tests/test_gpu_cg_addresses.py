"""The solver's kernels for arrays of 4 GiB and more (64-bit addresses) on small
grids: bitwise the fields and iteration counts of the 32-bit ones, for both
methods, alone and with the host-checked loop."""
import os

import numpy as np
import pytest

import oracle
import paper_2209_13768_gb300 as wfa
from test_gpu_cg_rows import FACES, _problem

pytestmark = pytest.mark.gpu


def _solve(p, dt, method, **env):
    os.environ.update(env)
    try:
        with wfa.Grid(p.shape, h=p.h) as g:
            g.set_bcs(p.bc)
            g.set_coeffs(p.k)
            g.set_field(p.T0)
            g.set_cg_method(method)
            it, res = g.implicit_step(dt, 2, rtol=1e-7, max_iter=300)
            return it, res, g.read_field()
    finally:
        for k in env:
            os.environ.pop(k, None)


@pytest.mark.parametrize("method", ["classic", "pipelined"])
@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("faces", range(len(FACES)))
@pytest.mark.parametrize("shape", [(37, 29, 23), (65, 17, 9), (130, 33, 20), (300, 4, 7), (130, 100, 40)])
def test_64_bit_addresses_are_bitwise_equal(shape, faces, kvar, method):
    p = _problem(faces, shape, kvar, seed=faces)
    k = p.k if np.isscalar(p.k) else np.asarray(p.k, dtype=np.float64)
    dt = 4.0 * oracle.dt_max(shape=p.shape, h=p.h, k=k, bc=p.bc)
    a = _solve(p, dt, method)
    for env in ({"WFA_CG_ADDR": "64"}, {"WFA_CG_ADDR": "64", "WFA_CG_LOOP": "host"}):
        b = _solve(p, dt, method, **env)
        assert a[:2] == b[:2]
        np.testing.assert_array_equal(a[2], b[2])
