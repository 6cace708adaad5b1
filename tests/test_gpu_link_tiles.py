"""Launches that change form with the number of tiles (1024 or 256 threads per
tile in linking, compression and loop properties; a block or a warp per tile in
the unions of tile-crossing edges; one or several parts per chain in the
operator scan and the record) against the oracle's roots and records, at the
sizes where the form changes."""
import numpy as np
import pytest

from test_gpu_parity import run_parity

pytestmark = pytest.mark.gpu

# tiles = L Q^2 ceil(beta / 16) / 128; the launches change above 304, at 2048
# (scan in parts), at 1024 (record in parts) and above 1216 (S = 1/2), 1824 (S = 1)
# and 3040 (a warp per tile for the crossing edges)
CASES = [
    (1216, 16.0 * 32, 1),      # 304 tiles: the last with 1024 threads per tile
    (1218, 16.0 * 32, 1),      # 305 tiles
    (304, 16.0 * 32, 2),       # 304 tiles, S = 1
    (306, 16.0 * 32, 2),       # 306 tiles
    (136, 16.0 * 32, 3),       # 306 tiles, S = 3/2
    (78, 16.0 * 32, 4),        # 312 tiles, S = 2
    (2, 16.0 * 64, 1),         # one tile, time blocks only
    (1520, 16.0 * 256, 1),     # 3040 tiles
    (1522, 16.0 * 256, 1),     # 3044 tiles
    (760, 16.0 * 128, 2),      # 3040 tiles, S = 1
    (762, 16.0 * 128, 2),      # 3048 tiles
    (608, 16.0 * 256, 1),      # 1216 tiles: the last block-per-tile launch of S = 1/2
    (610, 16.0 * 256, 1),      # 1220 tiles: the first warp-per-tile launch
    (456, 16.0 * 128, 2),      # 1824 tiles, S = 1: the last
    (458, 16.0 * 128, 2),      # 1832 tiles: the first
    (336, 16.0 * 128, 3),      # 3024 tiles, S = 3/2
    (338, 16.0 * 128, 3),      # 3042 tiles
    (2054, 16.0 * 256, 1),     # 4108 tiles: 4 scan parts, 8 record parts
    (80, 16.0 * 4, 3),         # S = 3/2: most edges cross
    (70, 16.0 * 4 + 3.0, 4),   # S = 2, ragged last window
]


@pytest.mark.parametrize("L,beta,Q", CASES)
def test_crossing_unions(L, beta, Q):
    run_parity(L, beta, Q=Q, seed=31 + L, nup=3)


def test_parts_in_an_uneven_batch():
    # a chain of several parts beside chains whose later parts are empty
    from paper_1810_07485_gb300 import lcqmc
    specs = [dict(L=2, beta=3.0, seed=1), dict(L=2054, beta=4096.0, seed=2), dict(L=34, beta=40.0, S=1.0, seed=3),
             dict(L=1030, beta=4096.0, seed=4), dict(L=6, beta=20.0, S=1.5, seed=5), dict(L=130, beta=7.0, S=2.0, seed=6)]
    b = lcqmc.Batch(specs)
    b.update(3)
    for i, sp in enumerate(specs):
        ch = lcqmc.Chain(sp["L"], sp["beta"], S=sp.get("S", 0.5), seed=sp["seed"])
        ch.update(3)
        assert np.array_equal(b.records(i), ch.records()), i
        ch.close()
    b.close()
