"""The depth pass with its CTAs far out of step: one works off a chain of a whole
chunk (1,024 transactions) while others run any number of chunks ahead."""
import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W
from tests.test_gpu_schemas import check, oe_pair

pytestmark = pytest.mark.gpu

CHUNK, N_WH, N_ITEMS = 1024, 4, 16


def order_statuses(n, seed):
    """Reads of warehouse 1's customers: transactions that wait for nothing."""
    rng = np.random.default_rng(seed)
    params = np.zeros((n, W.OE_PARAMS), np.int64)
    params[:, 0], params[:, 1], params[:, 2] = 1, rng.integers(0, 10, n), rng.integers(0, 3000, n)
    return {"ts": np.arange(n, dtype=np.int64), "type": np.full(n, G.T_OE_ORDER_STATUS, np.int32), "params": params,
            "P": W.OE_PARAMS}


def orders(bulk, at, w, item):
    """One-line new-orders of one customer, each waiting for the one before on
    several items, so that no chain of single waits shortens it."""
    bulk["type"][at] = G.T_OE_NEW_ORDER
    bulk["params"][at] = 0
    bulk["params"][at, 0], bulk["params"][at, 3] = w, 1
    bulk["params"][at, 4] = item | w << 24 | 1 << 40


def ahead_of_the_source():
    """Chunk 129 waits for chunk 128, whose CTA is still in chunk 0."""
    bulk = order_statuses(130 * CHUNK, 1)
    orders(bulk, np.arange(1, CHUNK), 0, 0)
    orders(bulk, np.r_[127 * CHUNK:128 * CHUNK + 1, 129 * CHUNK:130 * CHUNK], 2, 1)
    return bulk, 2 * CHUNK


def behind_the_source(chunks):
    """In chunk 1 a payment waits for two reads of its customer: first for the
    later one, behind the chain of the chunk's orders, then for the one in chunk
    0, whose CTA is at the bulk's end by then."""
    bulk = order_statuses(chunks * CHUNK, 2)
    orders(bulk, np.arange(CHUNK, 2 * CHUNK - 2), 0, 0)
    bulk["params"][[0, 2 * CHUNK - 2, 2 * CHUNK - 1], :3] = 0
    bulk["type"][2 * CHUNK - 1] = G.T_OE_PAYMENT
    bulk["params"][2 * CHUNK - 1, 3] = 5
    return bulk, CHUNK


@pytest.mark.parametrize("launch", [0, 1])
@pytest.mark.parametrize("build", [ahead_of_the_source, lambda: behind_the_source(72), lambda: behind_the_source(120),
                                   lambda: behind_the_source(200)], ids=["ahead", "72", "120", "200"])
def test_ctas_out_of_step(build, launch):
    bulk, depth = build()
    g, o = oe_pair(N_WH, N_ITEMS, max_bulk=1 << 18)
    obj, cls, root = o.extract(bulk, G.CONFLICT_PAPER, oracle.MAX_OPS)
    expect = oracle.graph_stats(oracle.levels(obj, cls, o.num_objects()), root)
    assert expect[0] == depth
    b = g.submit_dict(bulk).execute("kset", kset_launch=launch)
    stats = b.sync()
    st, out = b.results()
    b.free()
    assert (stats["depth"], stats["w0"], stats["cross"]) == expect
    ost, oout = o.execute(bulk, R=g.width)
    check(g, o, st, out, ost, oout, oe=True)
    g.close()
