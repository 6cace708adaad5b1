"""Record read-back: the records that come back staged behind the updates equal
the ones read in other portions, at the staging buffer's and the ring's edges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,max_n", [(1, 1 << 16), (255, 1 << 16), (256, 1 << 16), (257, 1 << 16),
                                     (300, 7), (4096, 1 << 16), (4100, 4097), (4100, 5)])
def test_records_in_any_portions(n, max_n):
    from paper_1810_07485_gb300 import lcqmc
    L, beta, seed = 4, 2.0, 9
    a, b = lcqmc.Chain(L, beta, seed=seed), lcqmc.Chain(L, beta, seed=seed)
    try:
        want = []
        for k in range(0, n, 64):  # small portions, always below the staging buffer
            a.update(min(64, n - k))
            want.append(a.records())
        want = np.concatenate(want)
        assert len(want) == n
        b.update(n)
        got = [b.records(max_n)]
        while True:
            r = b.records(max_n)
            if not len(r):
                break
            got.append(r)
        got = np.concatenate(got)
        assert np.array_equal(got, want[-min(n, 4096):])
        assert len(b.records(0)) == 0
        b.update(2)  # the read position stays right afterwards
        a.update(2)
        assert np.array_equal(b.records(), a.records())
    finally:
        a.close()
        b.close()
