"""The device result arrays of a bulk that failed hold zeros, not what the
memory held before."""
import numpy as np
import pytest

import paper_1103_3105_gb300 as G
import workloads as W

pytestmark = pytest.mark.gpu


def device_words(torch, address, n):
    class View:
        __cuda_array_interface__ = {"shape": (n,), "typestr": "<i8", "version": 3, "data": (address, False)}
    return torch.as_tensor(View(), device="cuda").cpu().numpy().copy()


@pytest.mark.parametrize("strategy,mode", [("kset", 0), ("kset", 1), ("part", 0), ("part_relaxed", 0), ("scan", 0),
                                           ("auto", 0), ("tpl", 0), ("tpl_relaxed", 0)])
def test_invalid_debit_credit_bulk(strategy, mode):
    torch = pytest.importorskip("torch")
    n = 5000
    g = G.Database(dc=(4, 40, 4000), history_capacity=1 << 20, max_bulk=n)
    g.register(G.DC_TYPES)
    bulk = W.dc_bulk(n, 4000, 0.0, seed=3)
    for k in range(8):                     # every stream's memory has held results
        bulk["params"][:, 1] = 77
        b = g.submit_dict(bulk).execute(strategy, conflict_mode=mode)
        b.sync()
        b.free()
    bulk["params"][n // 2, 0] = 4000       # no such account
    for k in range(4):
        b = g.submit_dict(bulk).execute(strategy, conflict_mode=mode)
        try:
            with pytest.raises(G.GputxError) as e:
                b.sync()
            values = device_words(torch, G.gputx_bulk_results_device(b.h)[1], n)
        finally:
            b.free()
        assert e.value.status == G.EINVAL and not values.any()
    g.close()
