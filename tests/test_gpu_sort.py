"""The radix sort's shapes, reached through the strategies that group by it:
one CTA up to 4,096 pairs, tiles of 2,048 up to 2^19 and of 8,192 above, 8- and
10-bit digits.  Every result is a whole number, compared exactly."""
import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W

pytestmark = pytest.mark.gpu

EDGES = [2, 4095, 4096, 4097, 6144, 6145, (1 << 19), (1 << 19) + 1]


# branches: 8, 10 and 11 key bits (PART); accounts: 9 to 25 (SCAN)
@pytest.mark.parametrize("B,T,A", [(1, 1, 300), (200, 200, 40_000), (1000, 1000, 1_000_000), (1100, 1100, 22_000_000)])
@pytest.mark.parametrize("n", EDGES)
def test_sort_shapes(n, B, T, A):
    bulk = W.dc_bulk(n, A, 0.0, seed=n % 1000)
    want = None
    for strategy in ("part", "scan"):
        g = G.Database(dc=(B, T, A), history_capacity=n, max_bulk=n)
        g.register(G.DC_TYPES)
        b = g.submit_dict(bulk).execute(strategy)
        st, out = b.results()
        b.free()
        if want is None:
            want = oracle.OracleDB(dc=W.dc_tables(B, T, A), hist_cap=n).execute(bulk, 1)
        assert np.array_equal(st, want[0]) and np.array_equal(out, want[1]), strategy
        g.close()
