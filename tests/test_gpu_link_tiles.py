"""Launches that change form with the number of tiles (1024 or 256 threads per
tile in linking, compression and loop properties; a block or a warp per tile in
the unions of tile-crossing edges) against the oracle's roots and records, at
the sizes where the form changes."""
import pytest

from test_gpu_parity import run_parity

pytestmark = pytest.mark.gpu

# tiles = L Q^2 ceil(beta / 16) / 128; the launches change above 304 and 3040
CASES = [
    (1216, 16.0 * 32, 1),      # 304 tiles: the last with 1024 threads per tile
    (1218, 16.0 * 32, 1),      # 305 tiles
    (304, 16.0 * 32, 2),       # 304 tiles, S = 1
    (306, 16.0 * 32, 2),       # 306 tiles
    (136, 16.0 * 32, 3),       # 306 tiles, S = 3/2
    (78, 16.0 * 32, 4),        # 312 tiles, S = 2
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
