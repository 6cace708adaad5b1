"""Chains that outgrow the room reserved for them beside chains that do not, against
the oracle.  Two sites at low temperature hold 2 beta vertices and beta operators,
more than the reserve of any longer chain at these sizes: the vertices run out in
the insertion, which stops the update while the other spins' kernels run beside it;
the operators run out in the rewrite, behind the loop sums.  The update that stopped
is run again with the same keys after the buffers grew."""
import numpy as np
import pytest

from oracle import orc
from test_gpu_parity import assert_graph_equal, assert_records_equal, assert_state_equal, gpu_state
from test_gpu_server import _check_against_oracle, _wait

pytestmark = pytest.mark.gpu

VERTICES = dict(L=2, beta=8000.0, seed=5)    # grow at the fourth or fifth update
OPERATORS = dict(L=2, beta=45000.0, seed=5)  # vertices at the third update, operators at the sixth
# beside chains of every spin that stay within their reserve
OTHERS = [dict(L=64, beta=64.0, S=1.0, seed=2), dict(L=34, beta=40.0, S=1.5, seed=3),
          dict(L=20, beta=40.0, S=2.0, seed=4), dict(L=512, beta=100.0, seed=6)]


def oracle_records(sp, n):
    p = orc.params(sp["L"], sp["beta"], Q=int(2 * sp.get("S", 0.5)), seed=sp["seed"])
    return orc.keyed_run(p, 0, n, orc.neel(p))


def check(specs, n, grows):
    from paper_1810_07485_gb300 import lcqmc
    b = lcqmc.Batch(specs)
    b.set_temporal(True)
    b.update(n)
    for i, sp in enumerate(specs):
        got, want = b.records(i), oracle_records(sp, n)
        assert len(got) == n
        for t in range(n):
            assert_records_equal(got[t], want[t], (sp, t))
    b.close()
    for sp in specs[:grows]:  # these do outgrow their reserve
        ch = lcqmc.Chain(sp["L"], sp["beta"], seed=sp["seed"])
        ch.update(n)
        ch.sync()
        assert ch.geometry().replays > 0
        ch.close()


@pytest.mark.parametrize("between", [False, True])  # the growing chains ahead of the others, or between them
def test_vertices_run_out_beside_other_spins(between):
    grow = [VERTICES, dict(L=2, beta=9001.5, seed=8)]
    specs = [grow[0], *OTHERS[:2], grow[1], *OTHERS[2:]] if between else grow + OTHERS
    check(specs, 8, 1 if between else 2)


def test_operators_run_out_beside_short_chains():
    # every chain's rewrite adds up its own counts (at most 1024 tiles), one stops it
    check([OPERATORS, dict(OPERATORS, seed=9), dict(OPERATORS, beta=46001.0, seed=10)] + OTHERS
          + [dict(L=64, beta=16.0, seed=20 + i) for i in range(40)], 9, 1)


@pytest.mark.parametrize("beta,n", [(45000.0, 9), (1.1e6, 6)])  # 44 tiles; 1075, whose offsets are scanned ahead
def test_operators_run_out(beta, n):
    from paper_1810_07485_gb300 import lcqmc
    p = orc.params(2, beta, seed=5)
    st = orc.neel(p)
    ch = lcqmc.Chain(2, beta, seed=5)
    try:
        ch.set_temporal(True)
        grown = []
        for t in range(n):
            st, ro, go = orc.keyed_update(p, t, st, graph=t == n - 1)
            ch.update(1)
            assert_records_equal(ch.records()[0], ro, t)
            grown.append(int(ch.geometry().replays))
        assert_graph_equal(ch.export_graph(), go)
        assert_state_equal(gpu_state(ch), st)
        assert grown[-1] >= 2  # for its vertices, then for its operators
    finally:
        ch.close()


def test_served_chains_grow():
    from paper_1810_07485_gb300 import lcqmc
    mix = [dict(dict(S=0.5, n=9), **sp) for sp in [VERTICES, *OTHERS, OPERATORS]]
    srv = lcqmc.Server(hbm_budget=8 << 30, max_slots=4)
    tickets = [srv.submit(m["L"], m["beta"], m["n"], S=m["S"], seed=m["seed"]) for m in mix]
    res = _wait(srv, tickets)
    srv.close()
    for m, t in zip(mix, tickets):
        assert res[t].status == 0
        _check_against_oracle(res[t], m)


def test_many_chains_grow_at_different_updates():
    # 160 chains whose vertices reach the end of their reserve once in a few dozen
    # updates: one call stops at more updates than a fixed number of passes covers
    from paper_1810_07485_gb300 import lcqmc
    n, specs = 400, [dict(L=2, beta=3494.5 + i * 9.5 / 160, seed=100 + i) for i in range(160)]
    want, stops = [], set()
    for sp in specs:
        ch = lcqmc.Chain(sp["L"], sp["beta"], seed=sp["seed"])
        for t in range(n):
            ch.update(1)
            ch.sync()
            if ch.geometry().replays:
                stops.add(t)
                ch.update(n - t - 1)
                break
        want.append((list(ch.measure().sum), ch.records()[-256:]))  # a batch keeps 256 records a chain
        ch.close()
    assert len(stops) > 64
    b = lcqmc.Batch(specs)
    b.update(n)
    for i in range(len(specs)):
        assert list(b.measure(i).sum) == want[i][0] and np.array_equal(b.records(i), want[i][1]), i
    b.close()
