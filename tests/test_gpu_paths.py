"""Debit-credit-only bulks executed path by path: windows of 256 positions over
groups by branch (K-SET under R/W, PART) and prefix sums by account (K-SET of
blind increments), at the windows' and slices' edges, with chains of repeated
accounts inside a window, across windows and across warps.  Whole numbers,
compared exactly with the oracle; d and w0 with the paths' lengths."""
import numpy as np
import pytest

import oracle
import paper_1103_3105_gb300 as G
import workloads as W

pytestmark = pytest.mark.gpu

B, T, A = 60, 120, 6000       # 100 accounts a branch


def accounts(pattern, n, rng):
    if pattern == "one account":
        return np.full(n, 4321)
    if pattern == "one branch":
        return 4300 + rng.integers(0, 100, n)
    if pattern == "pairs":          # neighbours and neighbours' neighbours share accounts
        return (np.arange(n) // 2 * 37 + np.arange(n) % 2 * (np.arange(n) % 3 == 0)) % A
    if pattern == "hot and rest":   # one long group among many short ones
        return np.where(rng.random(n) < 0.6, 17, rng.integers(0, A, n))
    return rng.integers(0, A, n)


@pytest.mark.parametrize("pattern", ["one account", "one branch", "pairs", "hot and rest", "uniform"])
@pytest.mark.parametrize("n", [1, 31, 33, 255, 256, 257, 513, 4097, 20_000, (1 << 20) + 1])
def test_paths(n, pattern):
    rng = np.random.default_rng(n)
    acct = accounts(pattern, n, rng)
    bulk = {"ts": np.arange(n, dtype=np.int64), "type": np.zeros(n, np.int32), "P": 2,
            "params": np.stack([acct, rng.integers(-(1 << 62), 1 << 62, n)], 1).astype(np.int64)}
    ost, oout = oracle.OracleDB(dc=W.dc_tables(B, T, A), hist_cap=n).execute(bulk, 1)
    for strategy, mode, size in (("kset", 0, 1), ("kset", 1, 1), ("part", 0, 1), ("part", 0, 7), ("scan", 0, 1)):
        g = G.Database(dc=(B, T, A), history_capacity=n, max_bulk=n)
        g.register(G.DC_TYPES)
        b = g.submit_dict(bulk).execute(strategy, conflict_mode=mode, part_size=size)
        stats = b.sync()
        st, out = b.results()
        b.free()
        assert np.array_equal(st, ost) and np.array_equal(out, oout), (strategy, mode, size)
        if strategy == "kset":
            lengths = np.bincount(acct if mode else acct // 100)
            assert (stats["depth"], stats["w0"]) == (lengths.max() - 1, (lengths > 0).sum())
        h = g.read(G.TBL_DC_HISTORY)
        assert np.array_equal(h[:, 0], bulk["ts"]) and np.array_equal(h[:, 4], bulk["params"][:, 1])
        with np.errstate(over="ignore"):
            want = np.zeros(T, np.int64)
            np.add.at(want, acct // 50, bulk["params"][:, 1])
        assert np.array_equal(g.read(G.TBL_DC_TELLER)[:, 0], want)
        g.close()


@pytest.mark.parametrize("P,shift", [(2, 0), (3, 0), (4, 0), (4, 1)])
def test_signature_widths_and_alignment(P, shift):
    """Rows of 2 and 4 parameters load as one 16-byte pair where their address
    allows it; of 3, or 8 bytes off, as two words."""
    torch = pytest.importorskip("torch")
    n = 3000
    rng = np.random.default_rng(P)
    params = rng.integers(0, 50, (n, P)).astype(np.int64)
    params[:, 0] = rng.integers(0, A, n)
    bulk = {"ts": np.arange(n, dtype=np.int64), "type": np.zeros(n, np.int32), "params": params, "P": P}
    ost, oout = oracle.OracleDB(dc=W.dc_tables(B, T, A), hist_cap=n).execute(bulk, 1)
    flat = torch.zeros(n * P + shift, dtype=torch.int64, device="cuda")
    flat[shift:] = torch.from_numpy(params.reshape(-1)).cuda()
    dev = flat[shift:].view(n, P)
    assert dev.data_ptr() % 16 == 8 * shift
    ts, ty = torch.arange(n, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for strategy in ("kset", "part", "scan"):
        g = G.Database(dc=(B, T, A), history_capacity=n, max_bulk=n)
        g.register(G.DC_TYPES)
        b = g.submit(ts, ty, dev).execute(strategy)
        st, out = b.results()
        b.free()
        assert np.array_equal(st, ost) and np.array_equal(out, oout), strategy
        g.close()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("pattern", ["one account", "one branch", "hot and rest", "pairs"])
@pytest.mark.parametrize("n", [127, 129, 130, 300, 8193])
def test_tpl_in_lock_order(n, pattern, mode):
    """Chains of up to 128 operations are served in timestamp order, longer
    ones in lock order: queues cut at a warp's and a CTA's 32 and 256."""
    rng = np.random.default_rng(n)
    acct = accounts(pattern, n, rng)
    bulk = {"ts": np.arange(n, dtype=np.int64), "type": np.zeros(n, np.int32), "P": 2,
            "params": np.stack([acct, rng.integers(-(1 << 62), 1 << 62, n)], 1).astype(np.int64)}
    ost, oout = oracle.OracleDB(dc=W.dc_tables(B, T, A), hist_cap=2 * n).execute(bulk, 1)
    g = G.Database(dc=(B, T, A), history_capacity=n, max_bulk=n)
    g.register(G.DC_TYPES)
    b = g.submit_dict(bulk).execute("tpl", conflict_mode=mode)
    st, out = b.results()
    b.free()
    assert np.array_equal(st, ost) and np.array_equal(out, oout)
    with np.errstate(over="ignore"):
        want = np.zeros(B, np.int64)
        np.add.at(want, acct // 100, bulk["params"][:, 1])
    assert np.array_equal(g.read(G.TBL_DC_BRANCH)[:, 0], want)
    g.close()


@pytest.mark.parametrize("n,n_br,block", [(150_000, 300, 0), (200_003, 1000, 0), (300_000, 70, 0), (300_000, 60, 1024),
                                          (160_001, 1, 0)])
def test_lock_order_in_runs(n, n_br, block):
    """More transactions than the grid holds 32 a warp: runs of several, chains
    that end in one, cross several or are too long a part of the bulk.  The
    balance after each transaction against its account's deltas summed up."""
    n_acc = 1000 * n_br
    bulk = W.dc_bulk(n, n_acc, 0.0, seed=n + n_br)
    g = G.Database(dc=(n_br, 10 * n_br, n_acc), history_capacity=n, max_bulk=n)
    g.register(G.DC_TYPES)
    b = g.submit_dict(bulk).execute("tpl", block_threads=block)
    b.sync()
    st, out = b.results()
    b.free()
    acc, delta = bulk["params"][:, 0], bulk["params"][:, 1]
    order = np.argsort(acc, kind="stable")
    run = np.cumsum(delta[order])
    first = np.searchsorted(acc[order], acc[order])
    expect = np.empty(n, np.int64)
    expect[order] = run - (run - delta[order])[first]
    want = np.zeros(n_acc, np.int64)
    np.add.at(want, acc, delta)
    assert not st.any() and np.array_equal(out[:, 0], expect)
    assert np.array_equal(g.read(G.TBL_DC_ACCOUNT)[:, 0], want)
    assert np.array_equal(g.read(G.TBL_DC_BRANCH)[:, 0], want.reshape(n_br, 1000).sum(1))
    g.close()
