"""The record of one long chain beside many short ones: every chain of a batch gets as
many parts as the launch allows for its number of chains."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("short", [40, 400, 2600])  # 8 parts (all of the long chain's), 6, one
def test_record_parts_by_number_of_chains(short):
    from paper_1810_07485_gb300 import lcqmc
    specs = [dict(L=2 + 2 * (i % 4), beta=1.0 + i % 7, S=0.5 + 0.5 * (i % 3), seed=i) for i in range(short)]
    specs.insert(short // 2, dict(L=2054, beta=4096.0, seed=99))  # 4108 tiles
    b = lcqmc.Batch(specs)
    b.update(3)
    for i in [0, 1, 2, short // 2 - 1, short // 2, short // 2 + 1, short]:
        sp = specs[i]
        ch = lcqmc.Chain(sp["L"], sp["beta"], S=sp.get("S", 0.5), seed=sp["seed"])
        ch.update(3)
        assert np.array_equal(b.records(i), ch.records()), i
        assert list(b.measure(i).sum) == list(ch.measure().sum), i
        ch.close()
    b.close()
