"""Order-entry bulks that do not end well: the order area overflows, or a wait
of the depth pass runs out.  The call says so, orders beyond the area leave no
trace, and what is reported of the graph is exact or unknown."""
import ctypes as C

import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W
from tests._helpers import gpu_logical_state, oracle_logical_state, states_equal
from tests.test_gpu_schemas import check, oe_pair

pytestmark = pytest.mark.gpu


def sync(b):
    """(status, stats) of a bulk that may have failed."""
    stats = G.ExecStats()
    return G.lib().gputx_sync_bulk(b.h, C.byref(stats)), stats


def test_depths_beside_an_execution_that_overflows():
    """The ranks and depths of a bulk of some thousand scan tiles are computed
    beside the execution, which fails for want of room while they are."""
    n, n_wh, n_items, fit = 1 << 20, 20, 2000, 1000
    g, o = oe_pair(n_wh, n_items, max_bulk=n, ord_cap=fit)
    next_id = g.read(G.TBL_OE_DISTRICT)[:, -1].sum()
    bulk = W.oe_bulk(n, n_wh, n_items=n_items, invalid_frac=0.0, seed=8, mix=(0.6, 0.3, 0.1))
    obj, cls, root = o.extract(bulk, G.CONFLICT_PAPER, oracle.MAX_OPS)
    expect = oracle.graph_stats(oracle.levels(obj, cls, o.num_objects()), root)
    b = g.submit_dict(bulk).execute("kset")
    status, stats = sync(b)
    b.free()
    assert status == G.ECAPACITY
    assert (stats.depth, stats.w0, stats.cross) == expect
    assert g.read(G.TBL_OE_DISTRICT)[:, -1].sum() - next_id == fit
    g.close()


@pytest.mark.parametrize("strategy,launch,types,batch", [("tpl", 0, G.OE_TYPES, False), ("kset", 1, G.OE_TYPES, False),
                                                         ("kset", 0, G.DC_TYPES + G.OE_TYPES, False),
                                                         ("kset", 1, G.DC_TYPES + G.OE_TYPES, False),
                                                         ("tpl", 0, G.OE_TYPES, True),
                                                         ("kset", 0, G.DC_TYPES + G.OE_TYPES, True)])
def test_orders_that_never_ran(strategy, launch, types, batch):
    """An order without room stops TPL and the level executors (one launch per
    level here).  The orders that they did not come to, most with slots past the
    area, are not completed: the index holds those that took an id, no others."""
    n, n_wh, n_items, fit = 30_000, 10, 200, 4000
    init = W.oe_tables(n_wh, n_items=n_items, seed=2)
    g = G.Database(dc=(1, 1, 1), oe=(n_wh, n_items), history_capacity=1, order_capacity=fit, orderline_capacity=15 * fit,
                   max_bulk=n)
    g.register(types)
    for t, rows in W.oe_rows(init).items():
        g.load(t, rows)
    bulk = W.oe_bulk(n, n_wh, n_items=n_items, invalid_frac=0.0, seed=4, mix=(0.8, 0.1, 0.1))
    if batch:
        bt = G.Batcher(g, tune=False, strategy=strategy, bulk_size=1 << 15, params_per_txn=W.OE_PARAMS)
        with pytest.raises(G.GputxError) as e:
            bt.run(bulk["ts"], bulk["type"], bulk["params"])
        status = e.value.status
        bt.close()
    else:
        b = g.submit_dict(bulk).execute(strategy, kset_launch=launch, narrow_max=1)
        status, _ = sync(b)
        b.free()
    assert status == G.ECAPACITY
    first, after = init["d_next_o_id"].reshape(-1), g.read(G.TBL_OE_DISTRICT)[:, -1]
    assert 0 < (after - first).sum() <= fit
    keys, rows = g.read_index(G.INDEX_ORDER)
    used = (keys != G.HKEY_EMPTY) & (keys != G.HKEY_TOMB)
    expect = [(d << 32) | i for d in range(10 * n_wh) for i in range(first[d], after[d])]
    assert np.array_equal(np.sort(keys[used]), np.array(expect, np.uint64))
    assert rows[used].max() < fit and len(np.unique(rows[used])) == used.sum()
    g.close()


@pytest.mark.parametrize("timing", [0, 1])
def test_depths_that_give_up(timing):
    """A 1 ns wait limit makes the depth pass give up in a chain of 680 orders
    (one tile for every scan and sort, so that nothing else waits).  Beside the
    execution that costs the depths alone; before it (timing) the bulk fails and
    nothing runs."""
    n, n_wh, n_items = 680, 1, 10
    g, o = oe_pair(n_wh, n_items, spin_limit_ns=1)
    params = np.zeros((n, W.OE_PARAMS), np.int64)
    params[:, 3], params[:, 4] = 1, 3 | 2 << 40
    bulk = {"ts": np.arange(n, dtype=np.int64), "type": np.full(n, G.T_OE_NEW_ORDER, np.int32), "params": params,
            "P": W.OE_PARAMS}
    b = g.submit_dict(bulk).execute("kset", timing=bool(timing))
    status, stats = sync(b)
    if timing:
        assert status == G.ETIMEOUT
        assert states_equal(gpu_logical_state(g, oe=True), oracle_logical_state(o))
    else:
        assert (status, stats.depth, stats.w0) == (G.OK, -1, -1)
        st, out = b.results()
        ost, oout = o.execute(bulk, R=g.width)
        check(g, o, st, out, ost, oout, oe=True)
    b.free()
    g.close()
