"""The device's forms of the two rounding steps of an imaginary time at the inputs a
random chain seldom meets: its tick count (one conversion instruction) at exact
halves, zero, denormals and the ends of the period, and a candidate's unit factor
with fewer than 33 significant bits.  Bit for bit against the oracle, whose forms are
the C library's ldexp, llrint and fma."""
import math

import numpy as np
import pytest

from oracle import orc
from test_gpu_parity import assert_graph_equal, assert_records_equal, assert_state_equal, gpu_state

pytestmark = pytest.mark.gpu


def edge_times(lo, hi, F):
    """Times in [lo, hi): every half tick k + 1/2 that a double holds, for small k from
    either end, with both neighbours; the ends; an even number of them."""
    t = {lo, np.nextafter(hi, lo), np.nextafter(lo, hi)}
    if lo == 0.0:
        t |= {5e-324, 2.0 ** -1023, np.nextafter(2.0 ** -1022, 0.0), 2.0 ** -1022, 2.0 ** -1022 * 1.5}
    ticks = 2.0 ** F
    for k in [0, 1, 2, 3, 4, 5, 1000, 1001, 2 ** 20, 2 ** 20 + 1]:
        for x in (lo + (k + 0.5) / ticks, hi - (k + 0.5) / ticks, lo + k / ticks):
            t |= {x, np.nextafter(x, 0.0), np.nextafter(x, math.inf)}
    t = np.array(sorted(x for x in t if lo <= x < hi))
    return t[: t.size // 2 * 2]


@pytest.mark.parametrize("L,beta,halves", [(4, 16.0, 6), (64, 64.0, 6), (512, 2048.0, 30)])
def test_tick_counts_at_the_edges(L, beta, halves):
    from paper_1810_07485_gb300 import lcqmc
    p = orc.params(L, beta, seed=3)
    st, g = orc.neel(p), orc.geometry(p)
    F = int(orc.keyed_run(p, 0, 1, orc.neel(p))[0]["F"])
    # even numbers of operators on bonds 0 and 2, whose sites share no other one
    cells = [np.zeros(0)] * g["ncell"]
    at = {(0, 0): edge_times(0.0, 16.0, F), (2, g["nwin"] - 1): edge_times(beta - 16.0, beta, F)}
    for (b, j), t in at.items():
        cells[orc.cell_index(p, b, j)] = t
    times = np.concatenate(cells)
    exact = [x for x in times if math.ldexp(x, F) % 1.0 == 0.5]  # ldexp is exact here
    assert len(exact) >= halves
    st = orc.State(st.s0, np.concatenate([[0], np.cumsum([len(c) for c in cells])]), times)
    ch = lcqmc.Chain(L, beta, seed=3)
    try:
        ch.set_temporal(True)
        ch.import_config(st.s0, st.op_ptr.astype(np.int32), st.op_tau, 7)
        for t in (7, 8):
            new, ro, go = orc.keyed_update(p, t, st, graph=True)
            ch.update(1)
            assert_records_equal(ch.records()[0], ro, (L, t))
            assert_graph_equal(ch.export_graph(), go, (L, t))
            assert_state_equal(gpu_state(ch), new, (L, t))
            st = new
    finally:
        ch.close()


# sweep, bond, window, draw of candidates of this chain and seed whose 53-bit draw is
# below 2^32, found by drawing the first 40000 sweeps
SMALL = [(14862, 3, 1, 0), (28414, 44, 0, 0), (6343, 55, 2, 1), (757, 22, 1, 2), (29052, 4, 0, 7), (10908, 28, 0, 12)]


@pytest.mark.parametrize("sweep,b,j,k", SMALL)
def test_unit_factor_of_small_draws(sweep, b, j, k):
    from paper_1810_07485_gb300 import lcqmc
    L, beta, seed = 64, 64.0, 1
    w = [int(x) for x in orc.philox([(1 << 24) | ((k + 1) // 2), b, j, sweep], [seed, 0])]
    u53 = ((w[0] | w[1] << 32) if k & 1 else (w[2] | w[3] << 32)) >> 11
    assert 0 < u53 < 2 ** 32
    p = orc.params(L, beta, seed=seed)
    st = orc.neel(p)
    ch = lcqmc.Chain(L, beta, seed=seed)
    try:
        ch.import_config(st.s0, st.op_ptr.astype(np.int32), st.op_tau, sweep)
        new, ro, go = orc.keyed_update(p, sweep, st, graph=True)  # every candidate of the Neel state is kept
        assert 16.0 * j + math.ldexp(u53, -49) in go["tau"]       # the window's start + 16 u53 2^-53
        ch.update(1)
        assert_graph_equal(ch.export_graph(), go)
        assert_state_equal(gpu_state(ch), new)
    finally:
        ch.close()
