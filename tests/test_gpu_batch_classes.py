"""Batches of per-cell-k grids without a periodic axis on both sides of the
choice between one and two steps a round, and rows too short for two: bitwise
the plain one-column kernel."""
import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa
from helpers import make_grid, run_gpu
from paper_2209_13768_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
@pytest.mark.parametrize("u", [(0.0, 0.0, 0.0), (0.2, -0.1, 0.05)])
@pytest.mark.parametrize("shape,count", [((204, 59, 15), 1), ((70, 73, 90), 13), ((109, 109, 4), 40), ((8, 90, 32), 60), ((7, 9, 8), 3)])
def test_batched_classes(shape, count, u, storage):
    rng = np.random.default_rng(count)
    probs = [W.Problem(shape=shape, T0=rng.uniform(0, 1, shape[::-1]).astype(np.float32),
                       k=np.exp(0.5 * rng.standard_normal(shape[::-1])).astype(np.float32), u=u, bc=[("dirichlet", 0.5)] * 6)
             for _ in range(3)]
    grids = [make_grid(probs[i % 3], storage=storage) for i in range(count)]
    for n in (5, 2):
        wfa.batch_run(grids, [n] * count)
    refs = [run_gpu(p, steps=7, storage=storage, variant=-1) for p in probs]
    for i in sorted({0, 1, 2, count - 1} & set(range(count))):
        np.testing.assert_array_equal(grids[i].read_field(), refs[i % 3])
    for g in grids:
        g.close()
