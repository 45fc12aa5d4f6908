"""Order-entry bulks that overflow the order area: the call reports ECAPACITY,
orders beyond the area leave no trace, and what is reported of the graph is
exact."""
import ctypes as C

import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W
from tests.test_gpu_schemas import oe_pair

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
