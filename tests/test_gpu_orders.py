"""Order-entry under K-SET: exact depths and levels from rounds over chunks of
1,024 transactions (chains inside a chunk, across chunks, runs of reads), levels
without the blind increments' edges, new-orders and order-statuses completed
after the levels.  Statuses, outputs, d, w0, c, the whole state and the index
against the oracle, exactly, in both launch forms."""
import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W
from tests.test_gpu_schemas import check, oe_pair

pytestmark = pytest.mark.gpu

ALL, PAY, READS, NO_PAY = (0.45, 0.43, 0.12), (0.02, 0.96, 0.02), (0.1, 0.1, 0.8), (0.6, 0.0, 0.4)


@pytest.mark.parametrize("launch", [0, 1])
@pytest.mark.parametrize("mode", [G.CONFLICT_PAPER, G.CONFLICT_ADD])
@pytest.mark.parametrize("n,n_wh,mix", [(1, 1, ALL), (1023, 1, ALL), (1024, 3, ALL), (1025, 3, PAY), (3000, 1, PAY),
                                        (5000, 2, READS), (4097, 1, READS), (9000, 3, NO_PAY), (30_000, 40, ALL)])
def test_levels_and_results(n, n_wh, mix, mode, launch):
    n_items = 300
    g, o = oe_pair(n_wh, n_items)
    ts0 = 0
    for k in range(2):      # the second bulk reads orders of the first
        bulk = W.oe_bulk(n, n_wh, n_items=n_items, remote_frac=0.1, invalid_frac=0.02, seed=900 + n + k, ts0=ts0,
                         mix=mix)
        if n_wh == 1:       # few customers: long runs of order-statuses, chains of orders
            bulk["params"][:, 2] %= 5
            bulk["params"][:, 1] %= 2
        ts0 += n
        obj, cls, root = o.extract(bulk, mode, oracle.MAX_OPS)
        lv = oracle.levels(obj, cls, o.num_objects())
        b = g.submit_dict(bulk).execute("kset", conflict_mode=mode, kset_launch=launch)
        stats = b.sync()
        st, out = b.results()
        b.free()
        ost, oout = o.execute(bulk, R=g.width)
        assert (stats["depth"], stats["w0"], stats["cross"]) == oracle.graph_stats(lv, root)
    check(g, o, st, out, ost, oout, oe=True)
    g.close()


def test_last_order_of_loaded_customers():
    """A customer loaded with a last order that has no row: every executor
    still looks it up and fails the bulk, as it did."""
    n_wh, n_items = 1, 50
    init = W.oe_tables(n_wh, n_items=n_items, seed=2)
    init["c_last_o_id"][7] = 3
    for strategy in ("kset", "tpl", "part"):
        g = G.Database(oe=(n_wh, n_items), order_capacity=100, orderline_capacity=1500, max_bulk=100)
        g.register(G.OE_TYPES)
        for t, rows in W.oe_rows(init).items():
            g.load(t, rows)
        p = np.zeros((1, 19), np.int64)
        p[0, 2] = 7
        b = g.submit(np.zeros(1, np.int64), np.full(1, G.T_OE_ORDER_STATUS, np.int32), p).execute(strategy)
        with pytest.raises(G.GputxError) as e:
            b.sync()
        assert e.value.status == G.EBOUNDS, strategy
        b.free()
        g.close()
