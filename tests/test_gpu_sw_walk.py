"""The Ising lattices on either side of the number of tiles from which the forest is
walked a second time (152 tiles of 64 x 32 sites), against the oracle."""
import pytest

from paper_1810_07485_gb300 import workloads
from test_gpu_sw import KC, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [512, 513])  # 128 and 153 tiles
def test_sw_parity_by_walk(L):
    run_parity(L, KC, seed=L, n=3, spins=workloads.ising_spins(L, seed=L))
