"""Unions of tile-crossing edges: both forms of the kernel (a block per tile for
few tiles, a warp per tile for many) against the oracle's roots and records, at
the sizes where the launch changes from one to the other."""
import pytest

from test_gpu_parity import run_parity

pytestmark = pytest.mark.gpu

# tiles = L Q^2 ceil(beta / 16) / 128; the launch changes above 3040
CASES = [
    (2, 16.0 * 64, 1),         # one tile, time blocks only
    (1520, 16.0 * 256, 1),     # 3040 tiles: the last block-per-tile launch
    (1522, 16.0 * 256, 1),     # 3044 tiles: the first warp-per-tile launch
    (760, 16.0 * 128, 2),      # 3040 tiles, S = 1
    (762, 16.0 * 128, 2),      # 3048 tiles
    (80, 16.0 * 4, 3),         # S = 3/2: most edges cross
    (70, 16.0 * 4 + 3.0, 4),   # S = 2, ragged last window
]


@pytest.mark.parametrize("L,beta,Q", CASES)
def test_crossing_unions(L, beta, Q):
    run_parity(L, beta, Q=Q, seed=31 + L, nup=3)
