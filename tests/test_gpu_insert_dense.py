"""Crowded cells: more operators than an insertion tile stages in shared
memory, more vertices than a warp's position marks hold, one cell with most of
them, a tile of more vertices than one pass of the operator rewrite takes
(8192), against the oracle (vertices, links, roots, new state, records)."""
import numpy as np
import pytest

from oracle import orc
from test_gpu_parity import assert_graph_equal, assert_records_equal, assert_state_equal, gpu_state

pytestmark = pytest.mark.gpu


def crowded(L, beta, Q, per_cell, only_bond, seed):
    """A valid state with `per_cell` operators (an even number) in every cell of
    the bonds that join the subspins 0 of sites 2k and 2k + 1 (of `only_bond`
    alone if it is given): each pair of spins flips together, no neighbour acts."""
    p = orc.params(L, beta, Q=Q, seed=seed)
    st = orc.neel(p)
    g = orc.geometry(p)
    rng = np.random.default_rng(seed)
    cells = [np.zeros(0)] * g["ncell"]
    for i in range(0, L, 2):
        b = i * Q * Q
        if only_bond is not None and b != only_bond:
            continue
        for j in range(g["nwin"]):
            t0, t1 = 16.0 * j, min(beta, 16.0 * (j + 1))
            cells[orc.cell_index(p, b, j)] = np.sort(rng.uniform(t0, t1, per_cell))
    ptr = np.concatenate([[0], np.cumsum([len(c) for c in cells])])
    return p, orc.State(st.s0, ptr, np.concatenate(cells))


@pytest.mark.parametrize("L,beta,Q,per_cell,only_bond", [
    (16, 20.0, 1, 40, None),    # marks exceeded in some warps only
    (16, 64.0, 1, 64, None),    # stage exceeded: neighbour operators from global memory
    (64, 40.0, 1, 20, None),
    (40, 64.0, 1, 400, 20),     # one bond holds every operator
    (2, 16.0, 1, 1000, None),
    (2, 16.0, 1, 9000, None),
    (12, 20.0, 2, 120, None),
    (6, 16.0, 3, 100, None),
    (4, 20.0, 4, 300, None),
])
def test_crowded_cells(L, beta, Q, per_cell, only_bond):
    from paper_1810_07485_gb300 import lcqmc
    p, st = crowded(L, beta, Q, per_cell, only_bond, seed=5)
    ch = lcqmc.Chain(L, beta, S=Q / 2, seed=5)
    try:
        ch.set_temporal(True)
        ch.import_config(st.s0, st.op_ptr.astype(np.int32), st.op_tau, 3)
        for t in range(3, 6):
            new, ro, go = orc.keyed_update(p, t, st, graph=True)
            ch.update(1)
            assert_records_equal(ch.records()[0], ro, (L, Q, t))
            assert_graph_equal(ch.export_graph(), go, (L, Q, t))
            assert_state_equal(gpu_state(ch), new, (L, Q, t))
            st = new
    finally:
        ch.close()
