"""The predictor with whole rows in a warp (nx <= 32): several rows a warp, rows
left over in y, lanes without a row, chunks of one to many layers; small grids
with tiled rows beside them.  Against the oracle (1e-12 relative L2, as the
other predictor tests)."""
import pytest

from tests import test_gpu_predictor_tiles as tt

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ywalls", [
    ((2, 3, 5), False), ((2, 20, 3), True), ((4, 9, 40), False), ((8, 5, 1), False), ((10, 9, 7), False),
    ((10, 8, 200), True), ((16, 1, 6), False), ((16, 6, 33), True), ((18, 15, 20), False), ((30, 27, 9), False),
    ((32, 32, 32), False), ((32, 30, 130), True), ((8, 64, 300), False), ((36, 3, 2), False), ((40, 40, 40), False),
    ((64, 64, 64), True), ((36, 30, 90), False)])
def test_whole_rows(dims, ywalls):
    tt.test_tiles_and_chunks(dims, ywalls)
