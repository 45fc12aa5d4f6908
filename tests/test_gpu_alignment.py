"""The batcher takes host arrays at any address."""
import numpy as np
import pytest

import paper_1103_3105_gb300 as G
import workloads as W
from tests.test_gpu_schemas import check, oe_pair

pytestmark = pytest.mark.gpu


def shifted(a, by):
    """A copy of `a` that starts `by` bytes off a multiple of 64."""
    raw = np.empty(a.nbytes + 128, np.uint8)
    at = -raw.ctypes.data % 64 + by
    out = raw[at:at + a.nbytes].view(a.dtype).reshape(a.shape)
    out[...] = a
    assert out.ctypes.data % 64 == by and np.ascontiguousarray(out, dtype=a.dtype) is out
    return out


@pytest.mark.parametrize("ts,type_,params", [(1, 0, 0), (4, 0, 0), (0, 1, 0), (0, 2, 0), (0, 0, 1), (0, 0, 4), (7, 3, 5),
                                             (8, 4, 8)])
def test_batcher_inputs_off_alignment(ts, type_, params):
    n, n_wh, n_items = 3000, 2, 50
    g, o = oe_pair(n_wh, n_items)
    bulk = W.oe_bulk(n, n_wh, n_items=n_items, seed=12)
    bt = G.Batcher(g, tune=False, strategy="kset", bulk_size=1 << 10, params_per_txn=W.OE_PARAMS)
    st, out = bt.run(shifted(bulk["ts"], ts), shifted(bulk["type"], type_), shifted(bulk["params"], params))
    ost, oout = o.execute(bulk, R=g.width)
    check(g, o, st, out, ost, oout, oe=True)
    bt.close()
    g.close()
