"""Swendsen-Wang launches that change form with the number of 64 x 32 tiles
(1024 or 256 threads per tile above 304; no second walk of the forest above
2048; graphs of eight updates and of one), against the oracle."""
import numpy as np
import pytest

from oracle import orc
from paper_1810_07485_gb300 import workloads
from test_gpu_sw import KC, assert_rec, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [768, 770, 2048, 2049])  # 288, 325, 2048, 2145 tiles
def test_sw_parity_by_tiles(L):
    run_parity(L, KC, seed=L, n=2, spins=workloads.ising_spins(L, seed=L))


def test_sw_blocks_of_updates():
    from paper_1810_07485_gb300 import lcqmc
    L, seed = 100, 6
    s = np.zeros(L * L, np.uint8)
    want = orc.sw_run(L, KC, seed, 0, 7 + 8 + 1 + 19, s)
    h = lcqmc.SWIsing(L, KC, seed=seed)
    try:
        for n in (7, 8, 1, 19):
            h.update(n)
        got = h.records()
        assert len(got) == len(want)
        for t in range(len(want)):
            assert_rec(got[t], want[t], t)
        assert np.array_equal(h.spins(), s)
    finally:
        h.close()
