"""Order-entry under K-SET item by item: items whose operations end at, cross and
fill a warp's 32 positions, stock rows that wrap in long runs, several bulks in
one captured segment, depths across the chunks of the depth pass, and a bulk that overflows
the order area.  Against the oracle, exactly, and mixed with the executor that
walks the levels (kset_launch = 1)."""
import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W
from tests.test_gpu_schemas import check, oe_pair

pytestmark = pytest.mark.gpu

HOT = {"all": (0.45, 0.43, 0.12), "orders": (1.0, 0.0, 0.0), "payments": (0.0, 1.0, 0.0), "mixed": (0.1, 0.5, 0.4)}


def hot_bulk(n, n_wh, n_items, mix, seed, ts0=0):
    """Every stock row is hot; the customers are one, three or all of a district's."""
    bulk = W.oe_bulk(n, n_wh, n_items=n_items, remote_frac=0.1, invalid_frac=0.05, seed=seed, ts0=ts0, mix=HOT[mix])
    bulk["params"][:, 2] %= (1, 3, 3000)[seed % 3]
    bulk["params"][:, 1] %= 1 + seed % 2 * 9
    return bulk


@pytest.mark.parametrize("n,n_wh,mix", [(31, 1, "payments"), (32, 1, "payments"), (33, 1, "mixed"), (64, 1, "orders"),
                                        (65, 2, "all"), (500, 1, "orders"), (4000, 1, "mixed"), (20_000, 2, "all")])
def test_hot_items(n, n_wh, mix):
    n_items = 16
    g, o = oe_pair(n_wh, n_items)
    ts0 = 0
    for k, launch in enumerate((0, 1, 0, 0)):     # the level walk in between leaves the same state
        bulk = hot_bulk(n, n_wh, n_items, mix, n + k, ts0)
        ts0 += n
        b = g.submit_dict(bulk).execute("kset", kset_launch=launch)
        b.sync()
        st, out = b.results()
        b.free()
        ost, oout = o.execute(bulk, R=g.width)
        assert np.array_equal(st, ost) and np.array_equal(out, oout), (k, launch)
    check(g, o, st, out, ost, oout, oe=True)
    g.close()


@pytest.mark.parametrize("n,n_wh,mix", [(511, 1, "payments"), (1024, 1, "all"), (1025, 1, "mixed"), (8193, 2, "orders"),
                                        (9217, 1, "payments"), (140_000, 3, "all")])
def test_depths_across_chunks(n, n_wh, mix):
    """Chunks of 1,024, a ring of eight, tags that repeat after 128 chunks."""
    g, o = oe_pair(n_wh, 16, max_bulk=1 << 18)
    bulk = hot_bulk(n, n_wh, 16, mix, 11 + n)
    obj, cls, root = o.extract(bulk, G.CONFLICT_PAPER, oracle.MAX_OPS)
    lv = oracle.levels(obj, cls, o.num_objects())
    b = g.submit_dict(bulk).execute("kset")
    stats = b.sync()
    st, out = b.results()
    b.free()
    assert (stats["depth"], stats["w0"], stats["cross"]) == oracle.graph_stats(lv, root)
    ost, oout = o.execute(bulk, R=g.width)
    assert np.array_equal(st, ost) and np.array_equal(out, oout)
    g.close()


@pytest.mark.parametrize("sizes", [(1, 31, 33), (700, 1, 1, 299), (40,) * 63])
def test_bulks_of_a_segment(sizes):
    """An item's operations of all bulks of a captured segment run in one chain."""
    n_wh, n_items, n = 2, 16, sum(sizes)
    g, o = oe_pair(n_wh, n_items)
    bulk = hot_bulk(n, n_wh, n_items, "all", 7)
    bt = G.Batcher(g, tune=False, strategy="kset", bulk_size=1 << 12, params_per_txn=W.OE_PARAMS)
    st, out = bt.run_bulks(bulk["ts"], bulk["type"], bulk["params"], sizes)
    ost, oout = o.execute(bulk, R=g.width)
    check(g, o, st, out, ost, oout, oe=True)
    bt.close()
    g.close()


def test_orders_that_do_not_fit():
    """The bulk fails; orders beyond the area touched nothing, the others ran."""
    n_wh, n_items, n, fit = 1, 40, 300, 290
    g, _ = oe_pair(n_wh, n_items, ord_cap=fit)
    next_id, count = g.read(G.TBL_OE_DISTRICT)[:, -1].sum(), g.read(G.TBL_OE_STOCK)[:, -1].sum()
    bulk = W.oe_bulk(n, n_wh, n_items=n_items, invalid_frac=0.0, seed=3, mix=HOT["orders"])
    b = g.submit_dict(bulk).execute("kset")
    with pytest.raises(G.GputxError) as e:
        b.sync()
    assert e.value.status == G.ECAPACITY
    b.free()
    assert g.read(G.TBL_OE_DISTRICT)[:, -1].sum() - next_id == fit
    assert g.read(G.TBL_OE_STOCK)[:, -1].sum() - count == bulk["params"][:fit, 3].sum()
    g.close()
