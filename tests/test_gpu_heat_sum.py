"""total_heat against the exact sum, on fields whose range is wide and with
threads that add many blocks of cells.

Tolerance. Of a thread's fp64 sum every block of 16 cells (four groups of 4 of
one row) rounds once, by at most 2^-53 of sum |T|; the thread's parts, the 8
levels of a block's tree and the 12 roundings of the finish add at most 24 more
(the cell volume is 1). What the fp32 part rounds off is below 2^-66. The
fields that leave the fp32 range are added cell by cell: 16 roundings a block."""
import math
from fractions import Fraction

import numpy as np
import pytest

import paper_2209_13768_gb300 as wfa

pytestmark = pytest.mark.gpu

THREADS = 1216 * 256


def _bound(shape, adds=1):
    lanes = 32
    while lanes > 1 and 2 * lanes >= shape[0]:
        lanes //= 2
    rows_at_once = THREADS // lanes
    blocks = -(-shape[1] * shape[2] // rows_at_once) * -(-shape[0] // (16 * lanes))
    return (adds * blocks + 24) * 2.0 ** -53


def test_long_sums_keep_fp64():
    """A cell of 1, then 107 groups of small and tiny cells, for every thread:
    rounding errors of a group's parts that are lost at 2^-48 of the running sum
    all have the same sign, and add up to 1.8e-13."""
    n = 512
    v = [float.fromhex(x) for x in ("0x1.f9673p-13", "0x1.baf498p-38", "0x1.7e7792p-13", "0x1.fc158ep-37")]
    T = np.empty((n, n, n), np.float32)
    T[:] = np.tile(np.array(v, np.float32), n // 4)
    T.reshape(n * n, n)[:9728, :128:4] = 1.0   # the first group of every lane, rows of 8 a block
    ones = 9728 * 32
    exact = ones + (n ** 3 // 4) * sum(Fraction(x) for x in v) - ones * Fraction(v[0])
    with wfa.Grid((n, n, n)) as g:
        g.set_field(T)
        got = g.total_heat()
    assert abs(Fraction(got) - exact) <= Fraction(_bound((n, n, n))) * exact


@pytest.mark.parametrize("storage", [wfa.F32, wfa.BF16])
@pytest.mark.parametrize("shape", [(2, 700, 500), (3, 2, 2), (4, 900, 300), (5, 400, 90), (8, 300, 200), (9, 70, 60),
                                   (16, 301, 33), (17, 50, 40), (63, 40, 41), (64, 33, 30), (65, 41, 20), (127, 25, 30),
                                   (128, 30, 31), (129, 30, 30), (511, 20, 21), (516, 21, 20), (1030, 9, 41)])
def test_wide_ranges_and_row_lengths(shape, storage):
    rng = np.random.default_rng(shape[0])
    size = shape[::-1]
    fields = {
        "lognormal": np.exp(5.0 * rng.standard_normal(size)),
        "one large": np.where(np.arange(np.prod(size)).reshape(size) == 3, 1e8, rng.uniform(0, 1, size)),
        "signed": rng.uniform(-1, 1, size) * np.exp2(rng.integers(-60, 60, size)),
        "subnormal": rng.uniform(-1, 1, size) * 2.0 ** -140,
        "huge": np.where(rng.random(size) < 0.5, 3.0e38, -1.0),
    }
    with wfa.Grid(shape, storage=storage) as g:
        for name, T in fields.items():
            g.set_field(T.astype(np.float32))
            held = g.read_field().astype(np.float64).ravel()
            exact, mag = math.fsum(held), math.fsum(np.abs(held))
            assert abs(g.total_heat() - exact) <= _bound(shape, 16 if name == "huge" else 1) * mag + 2 ** -53 * abs(exact), name
