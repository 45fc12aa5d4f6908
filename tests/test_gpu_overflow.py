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
