"""The workloads on which this engine's speed is measured, each through the
public binding (``Database.submit`` / ``Bulk.execute`` / results, and the
batcher).

A case is one bulk (or one stream of bulks) of transactions over a loaded
database; a pass submits it, executes it and has its statuses and values.  A
pass changes the database as every bulk does: balances move, history, order
and call-forwarding rows are appended.  Appended rows go to areas of fixed
capacity; when the next pass would not fit, a fresh database takes over, as a
program that runs for long does it (the areas are sized so that this is rare).

``io``: "device" = signatures are CUDA tensors and the results stay on the
device (a client that produces and consumes on the GPU); "host" = pinned host
arrays in and out (the paper's boundary: transfers are part of the pass).

The relaxed strategies are not listed: their results depend on the order the
locks happened to be taken in, so two runs cannot be compared.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1103_3105_gb300 as G

# debit-credit database shapes: branches, tellers, accounts
DC_SIZES = {"tiny": (4, 40, 4_000), "odd": (37, 259, 289_303), "full": (1_000, 10_000, 10_000_000)}
N_SUB = 1_000_000          # subscribers (64 MB of rows and 400 MB of index: larger than L2)
SUB_CHILD_CAP = 32_000_000
OE_WH, OE_ITEMS, OE_DIST, OE_CUST, OE_LINES = 64, 100_000, 10, 3_000, 15
SUB_MIX = (0.30, 0.25, 0.25, 0.08, 0.08, 0.02, 0.02)
OE_MIX = (0.45, 0.43, 0.12)
OUT_WIDTH = {"dc": 1, "sub": 8, "oe": 4, "mix": 8}
PARAMS = {"dc": 2, "sub": 5, "oe": 4 + OE_LINES, "mix": 5}


def _case(name, schema, n, strategy, add=False, theta=0.0, io="device", db="full", via="bulk", pieces=1):
    return {"name": name, "schema": schema, "n": n, "strategy": strategy, "add": add, "theta": theta, "io": io,
            "db": db, "via": via, "pieces": pieces}


def listed():
    return [
        # a served bulk: 1 ms of arrivals at 1 M transactions/s, host to host; launches and latency are all there is
        _case("dc_auto_1000_host", "dc", 1_000, "auto", io="host"),
        # the repository's smallest configuration: 4 branches, so 4 chains about 1,000 k-sets deep
        _case("dc_kset_tiny", "dc", 4_096, "kset", db="tiny"),
        # an ordinary bulk of an uneven size by branch partitions, mildly skewed accounts
        _case("dc_part_200k", "dc", 200_003, "part", theta=0.5),
        # the benchmark's headline: one bulk of 2^22, k-sets under the paper's read/write model
        _case("dc_kset_4m", "dc", 1 << 22, "kset"),
        # the same bulk with the strategy left to the engine
        _case("dc_auto_4m", "dc", 1 << 22, "auto"),
        # blind increments: a shallow graph of wide k-sets, an uneven size
        _case("dc_kset_add_1m", "dc", 1_000_003, "kset", add=True, theta=0.5),
        # ordered locks over 1,000 branch counters
        _case("dc_tpl_1m", "dc", 1 << 20, "tpl"),
        # hot accounts: one branch's chain holds a large part of the bulk
        _case("dc_kset_hot_200k", "dc", 200_003, "kset", theta=0.99),
        # the subscriber mix: 80 % reads, inserts and deletes through the hash indexes
        _case("sub_kset_1m", "sub", 1 << 20, "kset"),
        # a served bulk of the mixed database: 1 ms at 20 M transactions/s, host to host
        _case("mix_kset_20k_host", "mix", 20_000, "kset", io="host"),
        # order-entry: transactions of up to 17 operations, deep graph, exact depths
        _case("oe_kset_200k", "oe", 200_003, "kset"),
        # a stream of uneven order-entry bulks through the batcher's captured graphs, host to host
        _case("oe_stream_130k_host", "oe", 130_001, "kset", io="host", via="batch", pieces=9),
    ]


def draw(rng):
    """One more case of the listed families: sizes log-uniform over each family's range, odd ones among them."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(("dc", "dc", "dc", "dc", "sub", "mix", "oe", "batch"))
    if family == "dc":
        strategy = rng.choice(("kset", "kset", "part", "tpl", "auto"))
        theta = rng.choice((0.0, 0.0, 0.5, 0.8, 0.99))
        db = rng.choice(("full", "full", "full", "odd", "tiny"))
        # deep chains cost by their length: few branches or hot accounts take smaller bulks
        hi = 1 << 22
        if strategy != "auto":
            if theta >= 0.8:
                hi = 200_000
            if db != "full":
                hi = min(hi, 100_000 if db == "odd" else 16_000)
        case = _case("", "dc", size(1_000, hi), strategy, add=rng.random() < 0.3, theta=theta,
                     io=rng.choice(("device", "device", "host")), db=db)
    elif family == "sub":
        theta = rng.choice((0.0, 0.8))
        case = _case("", "sub", size(4_000, 1 << 20 if theta == 0.0 else 200_000),
                     rng.choice(("kset", "part", "tpl", "auto")), theta=theta, io=rng.choice(("device", "host")))
    elif family == "mix":
        case = _case("", "mix", size(1_000, 200_000), "kset", theta=rng.choice((0.0, 0.8)), io="host")
    elif family == "oe":
        case = _case("", "oe", size(1_000, 200_000), rng.choice(("kset", "kset", "tpl")), add=rng.random() < 0.3)
    else:
        case = _case("", "oe", size(8_000, 130_000), "kset", io="host", via="batch", pieces=rng.randrange(1, 17))
    del case["name"]
    return case


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _zeta(n, theta):
    return float((torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** -theta).sum())


def _keys(g, n_keys, theta, size):
    """`size` keys of [0, n_keys): uniform, or Zipf(theta) (Gray et al.'s closed form) with the ranks spread over the
    keys by a fixed multiplication modulo n_keys, so that hot keys don't share a branch."""
    if theta == 0.0:
        return torch.randint(0, n_keys, (size,), generator=g, device="cuda")
    zetan, alpha = _zeta(n_keys, theta), 1.0 / (1.0 - theta)
    eta = (1.0 - (2.0 / n_keys) ** (1.0 - theta)) / (1.0 - (1.0 + 0.5 ** theta) / zetan)
    u = torch.rand(size, generator=g, device="cuda", dtype=torch.float64)
    r = (n_keys * (eta * u - eta + 1.0) ** alpha).long()
    r[u * zetan < 1.0 + 0.5 ** theta] = 1
    r[u * zetan < 1.0] = 0
    step = 0x9E3779B1
    while math.gcd(step, n_keys) != 1:
        step += 2
    return (r.clamp_(0, n_keys - 1) * (step % n_keys) + 12_345) % n_keys


def _dc_params(g, n, n_accounts, theta):
    delta = torch.randint(-99_999, 100_000, (n,), generator=g, device="cuda")
    return torch.stack([_keys(g, n_accounts, theta, n), delta], 1)


def _pick(g, n, mix):
    edges = torch.tensor(mix, dtype=torch.float64, device="cuda").cumsum(0)[:-1]
    return torch.bucketize(torch.rand(n, generator=g, device="cuda", dtype=torch.float64), edges)


def _sub_bulk(g, n, theta):
    def ri(lo, hi):
        return torch.randint(lo, hi, (n,), generator=g, device="cuda")

    type_ = _pick(g, n, SUB_MIX) + G.T_SUB_GET_SUBSCRIBER
    p = torch.zeros((n, 5), dtype=torch.int64, device="cuda")
    p[:, 0] = _keys(g, N_SUB, theta, n)
    kind, start, end = ri(1, 5), 8 * ri(0, 3), ri(1, 25)
    loc, bit, da, num = ri(0, 1 << 30), ri(0, 2), ri(0, 256), ri(0, 1 << 30)
    for t, cols in ((G.T_SUB_GET_ACCESS, (kind,)), (G.T_SUB_GET_NEW_DEST, (kind, start, end)),
                    (G.T_SUB_UPDATE_LOCATION, (loc,)), (G.T_SUB_UPDATE_FACILITY, (kind, bit, da)),
                    (G.T_SUB_INSERT_CF, (kind, start, start + 1 + end % 8, num)),
                    (G.T_SUB_DELETE_CF, (kind, start))):
        m = type_ == t
        for j, c in enumerate(cols):
            p[m, 1 + j] = c[m]
    return type_.int(), p


def _oe_bulk(g, n):
    """45 % new-orders of 5..15 distinct Zipf(0.8) items (1 % remote lines, 1 % with an unknown last item), 43 %
    payments, 12 % order-statuses."""
    def ri(lo, hi, *shape):
        return torch.randint(lo, hi, shape or (n,), generator=g, device="cuda")

    type_ = _pick(g, n, OE_MIX) + G.T_OE_NEW_ORDER
    p = torch.zeros((n, 4 + OE_LINES), dtype=torch.int64, device="cuda")
    p[:, 0], p[:, 1], p[:, 2] = ri(0, OE_WH), ri(0, OE_DIST), ri(0, OE_CUST)
    pay = type_ == G.T_OE_PAYMENT
    p[pay, 3] = ri(1, 5_001)[pay]
    no = type_ == G.T_OE_NEW_ORDER
    m = int(no.sum())
    # distinct items: 32 draws an order, sorted, the first of each value in front; the rare rest is filled up upwards
    cand = _keys(g, OE_ITEMS, 0.8, m * 32).reshape(m, 32).sort(1).values
    dup = torch.zeros_like(cand, dtype=torch.bool)
    dup[:, 1:] = cand[:, 1:] == cand[:, :-1]
    items = cand.gather(1, dup.to(torch.int8).sort(dim=1, stable=True).indices[:, :OE_LINES])
    for r in torch.nonzero((~dup).sum(1) < OE_LINES).flatten().tolist():
        u = torch.unique(cand[r])
        extra = [x for x in range(2 * OE_LINES) if x not in set(u.tolist())][:OE_LINES - len(u)]
        items[r] = torch.cat([u, torch.tensor(extra, dtype=torch.int64, device="cuda")])
    cnt = ri(5, OE_LINES + 1, m)
    bad = torch.rand(m, generator=g, device="cuda") < 0.01
    rows = torch.arange(m, device="cuda")
    items[rows[bad], cnt[bad] - 1] = OE_ITEMS
    w = p[no, 0][:, None]
    other = (w + ri(1, OE_WH, m, OE_LINES)) % OE_WH
    sw = torch.where(torch.rand((m, OE_LINES), generator=g, device="cuda") < 0.01, other, w)
    lines = items | (sw << 24) | (ri(1, 11, m, OE_LINES) << 40)
    lines[torch.arange(OE_LINES, device="cuda")[None, :] >= cnt[:, None]] = 0
    p[no] = torch.cat([p[no, :3], cnt[:, None], lines], 1)
    return type_.int(), p


def _bulk(case, seed):
    g = torch.Generator(device="cuda").manual_seed(1_103_000 + int(seed))
    n, schema, theta = case["n"], case["schema"], case["theta"]
    if schema == "dc":
        return torch.zeros(n, dtype=torch.int32, device="cuda"), _dc_params(g, n, DC_SIZES[case["db"]][2], theta)
    if schema == "sub":
        return _sub_bulk(g, n, theta)
    if schema == "oe":
        return _oe_bulk(g, n)
    type_, p = _sub_bulk(g, n, theta)      # half debit-credit, half subscriber, interleaved at random
    dc = torch.rand(n, generator=g, device="cuda") < 0.5
    type_[dc] = G.T_DC_DEBIT_CREDIT
    p[dc] = 0
    p[dc, :2] = _dc_params(g, n, DC_SIZES["full"][2], theta)[dc]
    return type_, p


# --------------------------------------------------------------------------
# the loaded databases (one fixed data set a schema; its rows are kept on the
# host, as a program keeps the data it loads)
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _sub_tables():
    rng = np.random.default_rng(1103)
    s = np.arange(N_SUB, dtype=np.int64)
    out = {G.TBL_SUB_SUBSCRIBER: rng.integers(0, 1 << 30, size=(N_SUB, 16), dtype=np.int64)}

    def children(universe, lowest):     # a non-empty (lowest = 1) random subset of `universe` per parent
        mask = rng.integers(lowest, 1 << universe, size=N_SUB)
        return np.nonzero((mask[:, None] >> np.arange(universe)) & 1)

    r, k = children(4, 1)
    out[G.TBL_SUB_ACCESS_INFO] = np.column_stack([s[r], k + 1, rng.integers(0, 1 << 30, size=(len(r), 4))])
    r, k = children(4, 1)
    m = len(r)
    out[G.TBL_SUB_SPECIAL_FACILITY] = np.column_stack(
        [s[r], k + 1, (rng.random(m) < 0.85).astype(np.int64), rng.integers(0, 256, size=(m, 2)),
         rng.integers(0, 1 << 30, size=m)])
    have = rng.integers(0, 8, size=m)
    f, st = np.nonzero((have[:, None] >> np.arange(3)) & 1)
    out[G.TBL_SUB_CALL_FORWARDING] = np.column_stack(
        [s[r[f]], k[f] + 1, 8 * st, 8 * st + rng.integers(1, 9, size=len(f)), rng.integers(0, 1 << 30, size=len(f))])
    return out


@functools.lru_cache(maxsize=None)
def _oe_tables():
    rng = np.random.default_rng(1104)
    nd, ns = OE_WH * OE_DIST, OE_WH * OE_ITEMS
    nc = nd * OE_CUST

    def rows(n, *cols):                 # a column is (lo, hi) at random or a constant
        t = np.zeros((n, len(cols)), dtype=np.int64)
        for j, c in enumerate(cols):
            t[:, j] = rng.integers(*c, size=n) if isinstance(c, tuple) else c
        return t

    return {G.TBL_OE_WAREHOUSE: rows(OE_WH, (0, 2_001), 0), G.TBL_OE_DISTRICT: rows(nd, (0, 2_001), 0, 1),
            G.TBL_OE_CUSTOMER: rows(nc, (0, 5_001), 0, 0, 0, 0), G.TBL_OE_ITEM: rows(OE_ITEMS, (100, 10_001)),
            G.TBL_OE_STOCK: rows(ns, (10, 101), 0, 0)}


def _open(case):
    """A loaded database and how many passes its append areas take."""
    n, schema = case["n"], case["schema"]
    kw, types, tables, passes = {"max_bulk": n}, [], {}, 1 << 40
    if schema in ("dc", "mix"):
        history = min(1_400_000_000, 20_000 * n)        # up to 56 GB of history rows
        kw.update(dc=DC_SIZES[case["db"]], history_capacity=history)
        types += G.DC_TYPES
        passes = min(passes, history // n)
    if schema in ("sub", "mix"):
        tables = _sub_tables()
        kw.update(sub=N_SUB, sub_child_capacity=SUB_CHILD_CAP)
        types += G.SUB_TYPES
        room = SUB_CHILD_CAP - len(tables[G.TBL_SUB_CALL_FORWARDING])
        passes = min(passes, int(room / (0.03 * n + 200)))     # 2 % of the transactions insert a row
    if schema == "oe":
        tables = _oe_tables()
        orders = min(40_000_000, 20_000 * n)
        kw.update(oe=(OE_WH, OE_ITEMS), order_capacity=orders, orderline_capacity=11 * orders)
        types += G.OE_TYPES
        passes = min(passes, int(orders / (0.5 * n + 200)))    # 45 % are new-orders of 10 lines on average
    db = G.Database(**kw)
    db.register(types)
    for table, rows in tables.items():
        db.load(table, rows)
    batcher = None
    if case["via"] == "batch":
        batcher = G.Batcher(db, tune=False, strategy=case["strategy"], bulk_size=1 << 16,
                            conflict_mode=int(case["add"]), params_per_txn=PARAMS[schema])
    return db, batcher, passes


def prepare(case, seed):
    type_, params = _bulk(case, seed)
    n, schema = case["n"], case["schema"]
    ts = torch.arange(n, dtype=torch.int64, device="cuda")
    s = {"case": case, "passes": 0}
    if case["io"] == "host":
        ts, type_, params = (x.cpu().pin_memory() for x in (ts, type_, params))
        s["status"] = torch.empty(n, dtype=torch.int32, pin_memory=True)
        s["values"] = torch.empty((n, OUT_WIDTH[schema]), dtype=torch.int64, pin_memory=True)
    if case["via"] == "batch":
        ts, type_, params = (x.numpy() for x in (ts, type_, params))
        # uneven bulks: shares 1, 2, 3, ... of the stream, the largest last
        k = case["pieces"]
        cuts = [n * i * (i + 1) // (k * (k + 1)) for i in range(k + 1)]
        s["sizes"] = [b - a for a, b in zip(cuts, cuts[1:])]
    s["in"] = (ts, type_, params.contiguous() if torch.is_tensor(params) else params)
    s["db"], s["batcher"], s["room"] = _open(case)
    torch.cuda.synchronize()
    return s


# --------------------------------------------------------------------------
# a pass
# --------------------------------------------------------------------------
class _DeviceArray:
    """A bulk's result array on the device (it keeps the bulk, whose memory it is)."""

    def __init__(self, bulk, address, shape, typestr):
        self.bulk = bulk
        self.__cuda_array_interface__ = {"shape": shape, "typestr": typestr, "data": (address, False), "version": 2}


def run(state):
    case = state["case"]
    if state["passes"] >= state["room"]:
        # full: a fresh database takes over (the old one goes with the last bulk that refers to it)
        state["db"] = state["batcher"] = None
        state["db"], state["batcher"], state["room"] = _open(case)
        state["passes"] = 0
    state["passes"] += 1
    db = state["db"]
    ts, type_, params = state["in"]
    if state["batcher"] is not None:
        return state["batcher"].run_bulks(ts, type_, params, state["sizes"])
    bulk = db.submit(ts, type_, params)
    bulk.execute(case["strategy"], conflict_mode=G.CONFLICT_ADD if case["add"] else G.CONFLICT_PAPER)
    if case["io"] == "host":
        out = bulk.results(state["status"], state["values"])
        bulk.free()
        return out
    bulk.sync()
    status, values = G.gputx_bulk_results_device(bulk.h)
    return (torch.as_tensor(_DeviceArray(bulk, status, (bulk.n,), "<i4"), device="cuda"),
            torch.as_tensor(_DeviceArray(bulk, values, (bulk.n, db.width), "<i8"), device="cuda"))


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    """Bytes of one pass: the signatures, statuses and values, and every cell that the procedures read or write once
    each (not whole sectors, and not what an analysis moves).  Operations: the additions."""
    n, schema = case["n"], case["schema"]
    io = n * (8 + 4 + 8 * PARAMS[schema] + 4 + 8 * OUT_WIDTH[schema])
    # an account read and written, a history row of five int64 fields
    dc = 16 + 40
    # by type: a row of 64 B; index entry + 16 B; two entries, a flag, up to three entries with end and number; ...
    sub = sum(f * b for f, b in zip(SUB_MIX, (64, 12 + 16, 12 + 4 + 1.5 * (12 + 8), 8, 12 + 8, 3 * 12 + 21, 2 * 12 + 1)))
    # new-order: district counter, rates, order row, index entry, customer, and per line (10) the item price, the stock
    # row's three fields read and written and the order line; payment: three customer cells and two totals, read and
    # written; order-status: two cells, an index entry, the order's count and first line, 10 amounts
    oe = sum(f * b for f, b in zip(OE_MIX, (16 + 24 + 33 + 12 + 8 + 10 * (8 + 32 + 20), 80, 16 + 12 + 12 + 80)))
    cells = {"dc": dc, "sub": sub, "oe": oe, "mix": (dc + sub) / 2}[schema]
    adds = {"dc": 3, "sub": 0, "oe": 20, "mix": 1.5}[schema]
    return {"bytes": io + n * cells, "flops": n * adds}


def exact(case, seed):
    """Debit-credit: every balance starts at zero, so a transaction's value is the sum of its account's deltas up to
    it.  The other schemas' procedures branch on what they read: no closed form."""
    if case["schema"] != "dc":
        return None
    _, params = _bulk(case, seed)
    a, d = params[:, 0].cpu().numpy(), params[:, 1].cpu().numpy()
    order = np.argsort(a, kind="stable")
    total = np.cumsum(d[order])
    head = np.r_[True, a[order][1:] != a[order][:-1]]
    start = np.maximum.accumulate(np.where(head, np.arange(len(a)), 0))
    values = np.empty(len(a), dtype=np.int64)
    values[order] = total - (total[start] - d[order][start])
    return np.zeros(len(a), dtype=np.int32), values.reshape(-1, 1)
