"""K-SET of single-operation bulks (subscriber types, alone and mixed with
debit-credit) run by run in windows of 512 sorted operations: runs and groups cut
at the windows' edges, one hot item, many items, every type in a round.
Statuses, outputs, d, w0 and the state against the oracle, exactly."""
import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W
from tests.test_gpu_schemas import check, sub_pair

pytestmark = pytest.mark.gpu

WRITES = (0.05, 0.05, 0.2, 0.2, 0.1, 0.2, 0.2)


@pytest.mark.parametrize("mix", [W.SUB_MIX, WRITES, (0.98, 0.0, 0.0, 0.02, 0.0, 0.0, 0.0)])
@pytest.mark.parametrize("n,n_sub", [(1, 1), (511, 1), (512, 1), (513, 3), (1025, 2), (3000, 1), (5000, 40),
                                     (20_000, 3000)])
def test_subscriber_rounds(n, n_sub, mix):
    g, o = sub_pair(n_sub, sub_child_capacity=1 << 16)
    ts0 = 0
    for k in range(2):
        bulk = W.sub_bulk(n, n_sub, 0.0, seed=40 + n + k, ts0=ts0, mix=mix)
        ts0 += n
        obj, cls, root = o.extract(bulk, 0, 1)
        lv = oracle.levels(obj, cls, o.num_objects())
        b = g.submit_dict(bulk).execute("kset")
        stats = b.sync()
        st, out = b.results()
        b.free()
        ost, oout = o.execute(bulk, R=g.width)
        assert (stats["depth"], stats["w0"]) == (lv.max(), (lv == 0).sum())
    check(g, o, st, out, ost, oout, sub=True, n_sub=n_sub)
    g.close()


@pytest.mark.parametrize("mode", [G.CONFLICT_PAPER, G.CONFLICT_ADD])
@pytest.mark.parametrize("n", [700, 9000])
def test_mixed_rounds(n, mode):
    B, T, A, n_sub = 3, 30, 900, 200
    init = W.sub_tables(n_sub, seed=3)
    g = G.Database(dc=(B, T, A), sub=n_sub, history_capacity=2 * n, sub_child_capacity=1 << 16, max_bulk=n)
    g.register(G.DC_TYPES + G.SUB_TYPES)
    for t, rows in W.sub_rows(init).items():
        g.load(t, rows)
    o = oracle.OracleDB(dc=W.dc_tables(B, T, A), sub=init, hist_cap=2 * n)
    parts = [W.dc_bulk(n, A, 0.5, seed=5), W.sub_bulk(n, n_sub, 0.5, seed=6, mix=WRITES)]
    bulk = W.concat_bulks(parts, np.random.default_rng(n).integers(0, 2, n))
    b = g.submit_dict(bulk).execute("kset", conflict_mode=mode)
    st, out = b.results()
    b.free()
    ost, oout = o.execute(bulk, R=g.width)
    check(g, o, st, out, ost, oout, dc=True, sub=True, n_sub=n_sub)
    g.close()
