"""The two-step passes (variant 7) against the plain one-column kernel (-1),
bitwise: at the edges of their 120-cell x tiles, 4- or 10-row tiles and z chunks, with
ragged rows and wrapped reads, and in sequences with the kernels that read
periodic copies, which it leaves stale."""
import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa
from helpers import make_grid, run_gpu
from paper_2209_13768_gb300 import workloads as W

pytestmark = pytest.mark.gpu

D, ZF, P = "dirichlet", "zeroflux", "periodic"
FACES = {
    "cold": [(D, 0.5), (D, -0.25), (D, 1.0), (D, 0.0), (D, 2.0), (D, 0.75)],
    "walls": [(ZF, 0.0)] * 6,
    "torus": [(P, 0.0)] * 6,
    "x": [(P, 0.0)] * 2 + [(D, 0.5), (ZF, 0.0), (ZF, 0.0), (D, 1.0)],
    "yz": [(D, 0.5), (ZF, 0.0)] + [(P, 0.0)] * 4,
}


def _problem(shape, faces, steps=6, seed=0, kvar=False, adv=True):
    rng = np.random.default_rng(seed)
    k = np.exp(0.5 * rng.standard_normal(shape[::-1])).astype(np.float32) if kvar else 0.8
    return W.Problem(shape=shape, T0=rng.uniform(0, 1, shape[::-1]).astype(np.float32), k=k,
                     u=tuple(rng.uniform(-0.4, 0.4, 3)) if adv else (0.0, 0.0, 0.0), bc=FACES[faces],
                     h=tuple(rng.uniform(0.8, 1.25, 3)), steps=steps)


@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
@pytest.mark.parametrize("kvar,adv", [(False, True), (True, False), (True, True)])
@pytest.mark.parametrize("faces", sorted(FACES))
@pytest.mark.parametrize("shape", [(8, 2, 2), (9, 3, 4), (64, 5, 7), (119, 4, 6), (120, 9, 5), (121, 8, 9), (124, 6, 8),
                                   (125, 13, 30), (240, 7, 5), (243, 10, 26), (245, 12, 11), (365, 21, 6)])
def test_pair_bitwise_at_tile_edges(shape, faces, kvar, adv, storage):
    p = _problem(shape, faces, kvar=kvar, adv=adv)
    ref = run_gpu(p, storage=storage, variant=-1)
    for zc in (0, 1, 3, 24):
        np.testing.assert_array_equal(run_gpu(p, storage=storage, depth=2, variant=7, zchunk=zc), ref, err_msg=f"zchunk {zc}")
    p.steps = 5
    np.testing.assert_array_equal(run_gpu(p, storage=storage, depth=2, variant=7), run_gpu(p, storage=storage, variant=-1))


@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("faces", ["torus", "x"])
def test_kernels_after_a_pair_pass_refresh_periodic_copies(faces, kvar):
    """Each of these reads periodic copies of the field a two-step pass wrote."""
    p = _problem((68, 11, 9), faces, kvar=kvar, adv=not kvar)
    ref = run_gpu(p, steps=8, variant=-1)
    for depth, variant in [(1, 3), (1, 5), (1, 6), (1, -1), (2, 1), (3, 2)]:
        with make_grid(p) as g:
            g.set_tuning(2, 7)
            g.step(4)
            g.set_tuning(depth, variant)
            g.step(4)
            np.testing.assert_array_equal(g.read_field(), ref, err_msg=f"variant {variant}")
    with make_grid(p) as g:   # the batched sweep
        g.set_tuning(2, 7)
        g.step(4)
        wfa.batch_run([g], [4])
        np.testing.assert_array_equal(g.read_field(), ref)
    p.u = (0.0, 0.0, 0.0)     # the implicit solver
    out = []
    for variant in (7, -1):
        with make_grid(p) as g:
            g.set_tuning(2 if variant == 7 else 1, variant)
            g.step(4)
            g.implicit_step(0.5, 2, rtol=1e-6)
            out.append(g.read_field())
    np.testing.assert_array_equal(out[0], out[1])


def test_faces_the_pair_pass_does_not_take():
    """Held layers, zero-flux walls with per-cell k and advection, and a bf16
    Dirichlet value the halo cannot hold run one step a pass."""
    held = W.Problem(shape=(40, 12, 10), T0=W.uniform01((40, 12, 10), 3), k=1.0, bc=[("dirichlet_cell", 0.5)] * 6, steps=5)
    np.testing.assert_array_equal(run_gpu(held, depth=2, variant=7), run_gpu(held, variant=-1))
    p = _problem((40, 12, 10), "cold")
    p.bc = [(D, 0.3)] * 6     # not a bf16 value
    np.testing.assert_array_equal(run_gpu(p, storage=wfa.BF16, depth=2, variant=7), run_gpu(p, storage=wfa.BF16, variant=-1))
    for p, storage in [(p, wfa.BF16), (_problem((40, 12, 10), "walls", kvar=True), wfa.F32), (held, wfa.F32)]:
        with make_grid(p, storage=storage) as g:
            g.set_tuning(2, 7)
            assert g.tuning()[0] == 1


@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
def test_batched_pairs_bitwise(storage):
    """Batched rounds of two steps (per-cell k) at odd and even counts, row
    widths on both sides of 8, 16 and 32 lanes a row, periodic axes and the
    short rows that keep single steps; then again from where they stopped."""
    probs = []
    for i, (shape, faces) in enumerate([((7, 9, 8), "cold"), ((8, 5, 6), "torus"), ((24, 50, 9), "x"), ((25, 20, 9), "x"),
                                        ((32, 47, 5), "walls"), ((33, 49, 12), "cold"), ((56, 24, 7), "torus"),
                                        ((64, 23, 70), "cold"), ((65, 12, 9), "yz"), ((128, 13, 6), "cold"),
                                        ((129, 12, 10), "walls"), ((131, 9, 8), "torus")]):
        adv = faces in ("cold", "torus") and i % 2 == 0
        probs.append(_problem(shape, faces, kvar=True, adv=adv, seed=i, steps=(i * 5) % 9 + (0 if i == 3 else 1)))
    grids = [make_grid(p, storage=storage) for p in probs]
    wfa.batch_run(grids, [p.steps for p in probs])
    for p, g in zip(probs, grids):
        np.testing.assert_array_equal(g.read_field(), run_gpu(p, storage=storage, variant=-1), err_msg=str(p.shape))
    wfa.batch_run(grids, [5] * len(grids))
    for p, g in zip(probs, grids):
        g.step(2)
        np.testing.assert_array_equal(g.read_field(), run_gpu(p, steps=p.steps + 7, storage=storage, variant=-1),
                                      err_msg=str(p.shape))
        g.close()
