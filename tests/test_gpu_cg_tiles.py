"""Classic CG over every tile that cg_dir / cg_res_u choose (64 x 16, 32 x 32 and
64 x 8 cells, 128 cells of few rows) against the oracle's iterates, on sizes
around each choice; tolerance as derived in test_gpu_cg_rows."""
import pytest

from test_gpu_cg_rows import FACES, _check, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kvar", [False, True])
@pytest.mark.parametrize("faces", range(len(FACES)))
@pytest.mark.parametrize("shape", [
    (66, 3, 20), (130, 4, 9), (257, 7, 12), (300, 8, 5), (64, 8, 11), (65, 9, 10),   # few rows: 32 lanes, 2 to 4 warps
    (70, 33, 20), (130, 20, 6), (200, 34, 4), (97, 64, 5),                           # 32 x 32
    (128, 17, 9), (60, 40, 7), (321, 24, 5), (64, 23, 6),                            # 64 x 8
    (64, 16, 17), (128, 32, 5)])                                                     # 64 x 16
def test_every_tile_matches_oracle(shape, faces, kvar):
    _check(_problem(faces, shape, kvar, seed=sum(shape) + 3 * faces))


def test_wide_grids_keep_tiles_whose_partials_fit():
    # 64 x 8 would fill better (200 rows), but 1094 x 25 tiles have more partials than there is room for
    _check(_problem(0, (70016, 200, 3), False, seed=1), m=2)
