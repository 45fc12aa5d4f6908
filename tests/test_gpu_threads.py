"""Databases of different sizes used from threads of their own."""
import threading

import numpy as np
import pytest

import paper_1103_3105_gb300 as G
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("strategy", ["kset", "part", "scan"])
def test_teller_and_branch_sums_of_two_databases(strategy):
    """The sums of 25,000 and of 8,000 cells gather in shared memory, 200 and 64
    KB, whichever thread launches first."""
    errors = []

    def work(shape, n, bulks):
        g = G.Database(dc=shape, history_capacity=n * bulks, max_bulk=n)
        try:
            g.register(G.DC_TYPES)
            bulk = W.dc_bulk(n, shape[2], 0.0, seed=n)
            for _ in range(bulks):
                b = g.submit_dict(bulk)
                try:
                    b.execute(strategy)
                    b.sync()
                finally:
                    b.free()
                bulk["ts"] = bulk["ts"] + n
            want = np.zeros(shape[1], np.int64)
            np.add.at(want, bulk["params"][:, 0] // (shape[2] // shape[1]), bulk["params"][:, 1])
            assert np.array_equal(g.read(G.TBL_DC_TELLER)[:, 0], bulks * want)
        except Exception as e:  # noqa: BLE001
            errors.append(e)
        finally:
            g.close()

    threads = [threading.Thread(target=work, args=a) for a in (((5000, 20_000, 100_000), 100_000, 60),
                                                               ((1000, 7000, 70_000), 40_000, 200))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
