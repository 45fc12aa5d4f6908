"""Order-entry databases that register some of its types only."""
import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W
from tests.test_gpu_schemas import check

pytestmark = pytest.mark.gpu

N_WH, N_ITEMS = 1, 50
TYPES = [(G.T_OE_ORDER_STATUS,), (G.T_OE_PAYMENT,), (G.T_OE_PAYMENT, G.T_OE_ORDER_STATUS)]


def database(types, init, n):
    g = G.Database(oe=(N_WH, N_ITEMS), order_capacity=100, orderline_capacity=1500, max_bulk=n)
    g.register(types)
    for t, rows in W.oe_rows(init).items():
        g.load(t, rows)
    return g


def run(g, bulk, how):
    if how == "batch":
        bt = G.Batcher(g, tune=False, strategy="kset", bulk_size=1 << 10, params_per_txn=W.OE_PARAMS)
        try:
            return bt.run(bulk["ts"], bulk["type"], bulk["params"])
        finally:
            bt.close()
    b = g.submit_dict(bulk).execute(how.rstrip("1"), kset_launch=int(how == "kset1"))
    try:
        b.sync()
        return b.results()
    finally:
        b.free()


@pytest.mark.parametrize("how", ["kset", "kset1", "tpl", "part", "auto", "batch"])
@pytest.mark.parametrize("types", TYPES)
def test_types_alone(types, how):
    n = 700
    init = W.oe_tables(N_WH, n_items=N_ITEMS, seed=2)
    bulk = W.oe_bulk(n, N_WH, n_items=N_ITEMS, seed=5, mix=(0, 0.6 * (G.T_OE_PAYMENT in types),
                                                           0.4 * (G.T_OE_ORDER_STATUS in types)))
    bulk["params"][:, 2] %= 20
    g = database(types, init, n)
    o = oracle.OracleDB(oe=init, ord_cap=100, ol_cap=1500, oid_cap=100)
    st, out = run(g, bulk, how)
    ost, oout = o.execute(bulk, R=g.width)
    check(g, o, st, out, ost, oout, oe=True)
    g.close()


@pytest.mark.parametrize("how", ["kset", "kset1", "tpl", "part", "auto", "batch"])
@pytest.mark.parametrize("types", TYPES[::2])
def test_last_order_without_a_row(types, how):
    """A customer loaded with a last order that has no row fails the bulk."""
    init = W.oe_tables(N_WH, n_items=N_ITEMS, seed=2)
    init["c_last_o_id"][7] = 3
    bulk = {"ts": np.zeros(1, np.int64), "type": np.full(1, G.T_OE_ORDER_STATUS, np.int32),
            "params": np.zeros((1, W.OE_PARAMS), np.int64), "P": W.OE_PARAMS}
    bulk["params"][0, 2] = 7
    g = database(types, init, 100)
    with pytest.raises(G.GputxError) as e:
        run(g, bulk, how)
    assert e.value.status == G.EBOUNDS
    g.close()
