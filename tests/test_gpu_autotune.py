"""The autotuner leaves alone what the launches do not use: launches of at most 304
tiles take 1024 threads per tile whatever is set, and the warps of the crossing-edge
unions count above 1216 tiles of spin 1/2 (1824 of spin 1) only.  The values set
before are none of the autotuner's own candidates."""
import pytest

pytestmark = pytest.mark.gpu

SET = dict(link_threads=256, link_x_warps=3, compress_threads=96)


@pytest.mark.parametrize("L,beta,S,link,link_x", [
    (64, 16.0, 0.5, False, False),      # one tile
    (1216, 512.0, 0.5, False, False),   # 304 tiles
    (1220, 512.0, 0.5, True, False),    # 305
    (4864, 512.0, 0.5, True, False),    # 1216
    (4868, 512.0, 0.5, True, True),     # 1217
    (1824, 512.0, 1.0, True, False),    # 1824
    (1826, 512.0, 1.0, True, True),     # 1826
])
def test_unused_sizes_keep_their_value(L, beta, S, link, link_x):
    from paper_1810_07485_gb300 import lcqmc
    ch = lcqmc.Chain(L, beta, S=S, seed=3)
    ch.set_tuning(**SET)
    t = ch.autotune(1)
    assert t == ch.tuning()
    assert t["link_threads"] in (128, 256) if link else t["link_threads"] == SET["link_threads"]
    assert t["link_x_warps"] in (2, 4, 8) if link_x else t["link_x_warps"] == SET["link_x_warps"]
    assert t["compress_threads"] in (64, 128) if link else t["compress_threads"] == SET["compress_threads"]
    assert ch.geometry().sweep == 8  # eight trials of one update all the same
    ch.close()


def test_batch_counts_each_spin():
    from paper_1810_07485_gb300 import lcqmc
    specs = [dict(L=2432, beta=512.0, seed=1), dict(L=2432, beta=512.0, S=1.0, seed=2)]  # 608 + 2432 tiles
    b = lcqmc.Batch(specs)
    b.set_tuning(**SET)
    t = b.autotune(1)
    assert t["link_x_warps"] in (2, 4, 8) and t["compress_threads"] in (64, 128)
    b.close()
