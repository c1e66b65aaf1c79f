"""Odd and even step counts in turn on periodic grids: a single step reads the
copies that the two-step passes before it left stale, alone and in batches.
Bitwise against the plain one-column kernel."""
import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa
from helpers import make_grid, run_gpu
from paper_2209_13768_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, ZF, P = "dirichlet", "zeroflux", "periodic"
FACES = {"torus": [(P, 0.0)] * 6, "x": [(P, 0.0)] * 2 + [(D, 0.5), (ZF, 0.0), (ZF, 0.0), (D, 1.0)],
         "yz": [(D, 0.5), (ZF, 0.0)] + [(P, 0.0)] * 4, "cold": [(D, 0.5)] * 6}
SHAPES = [(8, 2, 2), (9, 3, 2), (68, 11, 9), (70, 2, 13), (127, 12, 5)]


def _problem(shape, faces, kvar, seed):
    rng = np.random.default_rng(seed)
    k = np.exp(0.5 * rng.standard_normal(shape[::-1])).astype(np.float32) if kvar else 0.8
    return W.Problem(shape=shape, T0=rng.uniform(0, 1, shape[::-1]).astype(np.float32), k=k, u=(0.0, 0.0, 0.0), bc=FACES[faces])


@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("faces", ["torus", "x", "yz"])
@pytest.mark.parametrize("shape", SHAPES)
def test_odd_counts_after_two_step_passes(shape, faces, kvar, storage):
    p = _problem(shape, faces, kvar, 3)
    with make_grid(p, storage=storage, depth=2, variant=7) as g:
        done = 0
        for n in (2, 1, 4, 3, 3, 1, 2, 5):
            g.step(n)
            done += n
            np.testing.assert_array_equal(g.read_field(), run_gpu(p, steps=done, storage=storage, variant=-1), err_msg=f"after {done}")


@pytest.mark.parametrize("mode", ["rounds", "stream", "persistent"])
def test_odd_counts_in_batches(mode, monkeypatch):
    monkeypatch.setenv("WFA_BATCH_MODE", mode)
    cases = [(shape, faces, kvar, storage) for shape in SHAPES for faces in FACES for kvar in (False, True)
             for storage in (wfa.F32, wfa.BF16)]
    probs = [_problem(shape, faces, kvar, i) for i, (shape, faces, kvar, _) in enumerate(cases)]
    grids = [make_grid(p, storage=c[3]) for p, c in zip(probs, cases)]
    done = np.zeros(len(grids), int)
    for r in range(5):
        steps = [(3 * i + 5 * r + i // 7) % 6 for i in range(len(grids))]
        wfa.batch_run(grids, steps)
        done += steps
        if r in (1, 3):   # a two-step pass of its own in between
            for g in grids:
                g.set_tuning(2, 7)
                g.step(2)
            done += 2
    for p, c, g, n in zip(probs, cases, grids, done):
        np.testing.assert_array_equal(g.read_field(), run_gpu(p, steps=int(n), storage=c[3], variant=-1), err_msg=str(c))
        g.close()
