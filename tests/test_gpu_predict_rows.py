"""Prediction tiles whose row count is no power of two: row counts around them, last tiles that
end inside a 16-byte piece."""
import pytest

import test_gpu_predict_tiles as tiles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,F,depth", [(65_632, 33, 5), (65_633, 33, 8), (65_759, 36, 6), (65_920, 40, 8), (66_001, 48, 6),
                                       (65_663, 60, 8), (65_569, 80, 10), (65_791, 17, 4), (66_047, 16, 4)])
def test_rows(m, F, depth):
    tiles.test_tiles(m, F, depth, 0)
