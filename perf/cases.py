"""Workloads of the hash tables as a user's program runs them, for timing.

Every case is one kind of call sequence through the package's public entry
points (``Table``, ``BatchPlan``, ``Server``) on seeded synthetic data:

  lookup   one query batch against a resident table (device or pinned host keys)
  step     a batch of each operation on a resident table: insert a window of new
           keys, add to present keys, query present and absent keys, erase the
           window again (the table is as full after a pass as before it)
  build    build a table from nothing and probe it (the two sides of a join)
  groupby  sum values per key from nothing: upsert-add with Zipf keys, read back
  mixed    two op-coded batches (query / add / insert / erase) on one table, the
           second erasing what the first inserted and the other way round
  batched  many tables of uneven sizes, every operation, one plan launch
  serve    requests of uneven sizes against many tables, all queued at once

Two-choice and iceberg tables are filled to at most 0.85, where no insert can
fail: near 0.9 the key that finds both its buckets full depends on the order in
which concurrent inserts land.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2509_16407_gb300 as ws

DEVICE = "cuda"
ADD_MAX = 1000  # upsert-add values are uniform in [1, ADD_MAX]
DESIGNS = (("double", False), ("double", True), ("p2", False), ("p2", True), ("iceberg", True))


def listed():
    return [
        # a request handler looking up one user's worth of keys: launch latency
        {"name": "lookup_small", "kind": "lookup", "scheme": "double", "meta": True, "log2_slots": 20, "load": 0.75,
         "n": 1000, "hit": 0.9, "host": False},
        # a feature lookup whose keys arrive in page-locked host memory
        {"name": "lookup_host_2p24", "kind": "lookup", "scheme": "p2", "meta": True, "log2_slots": 24, "load": 0.8,
         "n": 3000001, "hit": 0.95, "host": True},
        # a dimension table of a small join
        {"name": "build_double_2p16", "kind": "build", "scheme": "double", "meta": False, "log2_slots": 16,
         "load": 0.7, "probe": 4.0, "hit": 0.5},
        # the build side of a large join, iceberg hashing
        {"name": "build_iceberg_2p23", "kind": "build", "scheme": "iceberg", "meta": True, "log2_slots": 23,
         "load": 0.8, "probe": 1.5, "hit": 0.5},
        # a table that L2 holds: every operation
        {"name": "step_p2m_2p22", "kind": "step", "scheme": "p2", "meta": True, "log2_slots": 22, "load": 0.85,
         "n": 1048577},
        # a table of a few gigabytes, batches that are small against it
        {"name": "step_doublem_2p26", "kind": "step", "scheme": "double", "meta": True, "log2_slots": 26,
         "load": 0.9, "n": 4194301},
        # the repository's benchmark: 2^28 slots, 2^24 operations of each class
        {"name": "step_double_2p28", "kind": "step", "scheme": "double", "meta": False, "log2_slots": 28,
         "load": 0.9, "n": 1 << 24},
        {"name": "step_p2_2p28", "kind": "step", "scheme": "p2", "meta": False, "log2_slots": 28, "load": 0.85,
         "n": 1 << 24},
        # aggregation of skewed rows (word counts, clicks per item)
        {"name": "groupby_zipf", "kind": "groupby", "scheme": "double", "meta": False, "log2_slots": 21,
         "load": 0.5, "n": 8000003, "theta": 0.99},
        # a key-value store under a skewed update-heavy load
        {"name": "mixed_zipf_2p27", "kind": "mixed", "scheme": "double", "meta": True, "log2_slots": 27,
         "load": 0.6, "n": 1 << 23, "theta": 0.99},
        # many uneven tables in one launch
        {"name": "batched_1024", "kind": "batched", "scheme": "double", "meta": False, "tables": 1024,
         "log2_min": 10, "log2_max": 22, "ops_min": 1 << 8, "ops_max": 1 << 19, "sizes": 4},
        # a request server over many tables, pinned request buffers
        {"name": "serve_32", "kind": "serve", "scheme": "double", "meta": False, "tables": 32, "log2_min": 16,
         "log2_max": 22, "requests": 96, "ops_max": 1 << 17, "sizes": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lookup", "lookup", "step", "step", "step", "build", "build", "groupby", "mixed", "batched",
                       "serve"])
    scheme, meta = rng.choice(DESIGNS)
    top = 0.9 if scheme == "double" else 0.85
    c = {"kind": kind, "scheme": scheme, "meta": meta}
    if kind == "lookup":
        c.update(log2_slots=rng.randint(14, 28), load=round(rng.uniform(0.4, top), 3), n=_log_int(rng, 1, 1 << 24),
                 hit=round(rng.uniform(0, 1), 2), host=rng.random() < 0.25)
    elif kind == "step":
        b = rng.randint(14, 27)
        c.update(log2_slots=b, load=round(rng.uniform(0.5, top), 3), n=_log_int(rng, 256, min(1 << 24, 4 << b)))
    elif kind == "build":
        c.update(log2_slots=rng.randint(12, 25), load=round(rng.uniform(0.3, top), 3),
                 probe=round(rng.uniform(0.2, 4), 2), hit=round(rng.uniform(0, 1), 2))
    elif kind == "groupby":
        c.update(log2_slots=rng.randint(14, 24), load=round(rng.uniform(0.2, 0.6), 3),
                 n=_log_int(rng, 10000, 1 << 24), theta=round(rng.uniform(0.5, 1.1), 2))
    elif kind == "mixed":
        c.update(log2_slots=rng.randint(18, 26), load=round(rng.uniform(0.4, 0.7), 3),
                 n=_log_int(rng, 1000, 1 << 23), theta=round(rng.uniform(0.5, 1.1), 2))
    elif kind == "batched":
        c.update(tables=_log_int(rng, 8, 512), log2_min=10, log2_max=rng.randint(14, 22), ops_min=1 << 8,
                 ops_max=_log_int(rng, 1 << 12, 1 << 19), sizes=rng.randint(0, 1 << 20))
    else:
        c.update(tables=rng.randint(4, 32), log2_min=14, log2_max=rng.randint(17, 22),
                 requests=_log_int(rng, 8, 96), ops_max=_log_int(rng, 1 << 10, 1 << 17), sizes=rng.randint(0, 1 << 20))
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _s64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


def _mix(z):
    """The splitmix64 finaliser on int64 tensors (a bijection)."""
    for sh, m in ((30, 0xBF58476D1CE4E5B9), (27, 0x94D049BB133111EB)):
        z = (z ^ ((z >> sh) & ((1 << (64 - sh)) - 1))) * _s64(m)
    return z ^ ((z >> 31) & ((1 << 33) - 1))


def _keys(seed, start, n):
    """Keys start .. start + n - 1 of the splitmix64 stream of the seed: distinct."""
    i = torch.arange(start + 1, start + n + 1, dtype=torch.int64, device=DEVICE)
    return _mix(i * _s64(0x9E3779B97F4A7C15) + _s64(seed * 0xD1342543DE82EF95 + 1))


def _gen(seed, what):
    return torch.Generator(device=DEVICE).manual_seed((int(seed) * 1000003 + what) % (1 << 62))


def _index(seed, what, n, bound):
    return torch.randint(0, max(1, bound), (n,), generator=_gen(seed, what), dtype=torch.int64, device=DEVICE)


def _zipf(seed, what, n, bound, theta):
    """Indices in [0, bound): item k has about Zipf(theta) mass (continuous inverse)."""
    u = torch.rand(n, generator=_gen(seed, what), dtype=torch.float64, device=DEVICE)
    if abs(theta - 1.0) < 1e-9:
        x = torch.exp(u * math.log(bound + 1))
    else:
        e = 1.0 - theta
        x = (u * ((bound + 1) ** e - 1.0) + 1.0) ** (1.0 / e)
    return (x.to(torch.int64) - 1).clamp_(0, bound - 1)


def _values(keys):
    return keys * 3


def _hits(seed, what, n, present, hit):
    """Stream positions of n lookups: a share `hit` among the first `present`, the rest beyond 2^40."""
    i = _index(seed, what, n, present)
    miss = torch.rand(n, generator=_gen(seed, what + 1), device=DEVICE) >= hit
    return torch.where(miss, i + (1 << 40), i), miss


def _at(seed, pos):
    """Keys at given stream positions."""
    return _mix((pos + 1) * _s64(0x9E3779B97F4A7C15) + _s64(seed * 0xD1342543DE82EF95 + 1))


def _slots(c):
    return 1 << c["log2_slots"]


def _counts(c):
    """(keys resident all the time, window of keys inserted and erased in a pass)."""
    s = _slots(c)
    if c["kind"] == "step":
        w = max(1, int(0.05 * s))
        return int(c["load"] * s) - w, w
    return max(1, int(c["load"] * s)), 0


def _inputs(c, seed):
    """The batches of one pass, and for exact() the indices behind them."""
    p, w = _counts(c)
    d = {}
    if c["kind"] == "lookup":
        pos, d["miss"] = _hits(seed, 11, c["n"], p, c["hit"])
        d["q"] = _at(seed, pos)
    elif c["kind"] == "step":
        n = c["n"]
        d["wk"] = _keys(seed, p, w)
        d["ui"], d["qi"] = _index(seed, 21, n, p), _index(seed, 22, n, p)
        d["uk"], d["qk"] = _at(seed, d["ui"]), _at(seed, d["qi"])
        d["uv"] = _index(seed, 23, n, ADD_MAX) + 1
        d["ak"] = _keys(seed, 1 << 40, n)
    elif c["kind"] == "build":
        d["k"] = _keys(seed, 0, p)
        pos, d["miss"] = _hits(seed, 31, max(1, int(c["probe"] * p)), p, c["hit"])
        d["q"] = _at(seed, pos)
    elif c["kind"] == "groupby":
        d["gi"] = _zipf(seed, 41, c["n"], p, c["theta"])
        d["k"], d["v"] = _at(seed, d["gi"]), _index(seed, 42, c["n"], ADD_MAX) + 1
        d["g"] = _keys(seed, 0, p)
    return d


def _mixed_pair(seed, n, present, window, theta):
    """Two op-coded batches of n ops: 50% query and 40% add of present keys (Zipf, the queried and the added keys
    disjoint), 5% insert and 5% erase of distinct window keys; the second batch swaps the inserted and erased keys."""
    m = max(1, min(n // 20, window))
    out = []
    for half in (0, 1):
        i = _zipf(seed, 51 + half, n, present, theta)
        ops = torch.where(i % 9 < 5, ws.MX_QUERY, ws.MX_ADD).to(torch.uint8)
        keys = _at(seed, i)
        at = torch.randperm(n, generator=_gen(seed, 53 + half), device=DEVICE)[: 2 * m]
        win = _keys(seed, present, 2 * m)
        ins = half == 0
        ops[at[:m]] = ws.MX_INSERT if ins else ws.MX_ERASE
        ops[at[m: 2 * m]] = ws.MX_ERASE if ins else ws.MX_INSERT
        k = min(m, max(0, n - m))
        keys[at[:m]] = win[:m]
        keys[at[m: m + k]] = win[m: m + k]
        vals = torch.where(ops == ws.MX_INSERT, _values(keys), _index(seed, 55 + half, n, ADD_MAX) + 1)
        vals = torch.where((ops == ws.MX_QUERY) | (ops == ws.MX_ERASE), torch.zeros_like(vals), vals)
        out.append((ops, keys, vals))
    return out, m


def _fill(t, seed, count, start=0, chunk=1 << 25):
    for a in range(0, count, chunk):
        k = _keys(seed, start + a, min(chunk, count - a))
        t.insert(k, _values(k))


def _table(c, slots):
    return ws.Table(slots, c["scheme"], c["meta"])


def _sizes(c, what, count, lo, hi):
    """Sizes log-uniform in [lo, hi): the case's own, the same for every seed."""
    r = np.random.RandomState(c["sizes"] * 31 + what)
    return np.exp2(r.uniform(math.log2(lo), math.log2(hi), count)).astype(np.int64)


# ---------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c = case
    if c["kind"] == "batched":
        return _prepare_batched(c, seed)
    if c["kind"] == "serve":
        return _prepare_serve(c, seed)
    t = _table(c, _slots(c))
    s = {"case": c, "table": t}
    p, _ = _counts(c)
    if c["kind"] == "mixed":
        pair, m = _mixed_pair(seed, c["n"], p, int(0.05 * _slots(c)), c["theta"])
        _fill(t, seed, p)
        _fill(t, seed, m, start=p + m)  # the first batch erases these and inserts the m keys before them
        s["pair"] = pair
        return s
    if c["kind"] in ("lookup", "step"):
        _fill(t, seed, p)
    s.update({k: v for k, v in _inputs(c, seed).items() if k not in ("miss", "ui", "qi", "gi")})
    if c["kind"] == "step":
        s["wv"] = _values(s["wk"])
    elif c["kind"] == "build":
        s["v"] = _values(s["k"])
    elif c.get("host"):
        s["q"] = s["q"].cpu().pin_memory()
    return s


def run(state):
    c = state["case"]
    if c["kind"] == "batched":
        state["plan"].launch()
        return state["out"]
    if c["kind"] == "serve":
        return _run_serve(state)
    t = state["table"]
    if c["kind"] == "lookup":
        v, st = t.query(state["q"], return_status=True)
        return {"values": v, "status": st}
    if c["kind"] == "step":
        ins = t.insert(state["wk"], state["wv"], return_status=True)
        up = t.upsert(state["uk"], state["uv"], op="add", return_status=True)
        pos = t.query(state["qk"])
        neg, neg_st = t.query(state["ak"], return_status=True)
        ev, est = t.erase(state["wk"], return_values=True, return_status=True)
        return {"insert": ins, "upsert": up, "present": pos, "absent": neg, "absent_status": neg_st, "erased": ev,
                "erase_status": est}
    if c["kind"] == "build":
        t.clear()
        st = t.insert(state["k"], state["v"], return_status=True)
        v, q = t.query(state["q"], return_status=True)
        return {"insert": st, "values": v, "status": q}
    if c["kind"] == "groupby":
        t.clear()
        t.upsert(state["k"], state["v"], op="add")
        v, st = t.query(state["g"], return_status=True)
        return {"sums": v, "status": st}
    return [t.mixed(ops, keys, vals) for ops, keys, vals in state["pair"]]


def _prepare_batched(c, seed):
    T = c["tables"]
    caps = 1 << np.floor(np.log2(_sizes(c, 61, T, 1 << c["log2_min"], 1 << c["log2_max"]))).astype(np.int64)
    nops = _sizes(c, 62, T, c["ops_min"], c["ops_max"])
    fill = (0.75 * caps).astype(np.int64)
    win = np.maximum(1, np.minimum(nops // 8, caps // 20))
    nq, nu = np.maximum(1, nops // 2), np.maximum(1, nops * 3 // 8)
    # one stream of keys, table by table: resident, then window
    start = np.concatenate([[0], np.cumsum(fill + win)])
    tot_q, tot_u, tot_w = int(nq.sum()), int(nu.sum()), int(win.sum())

    def per_table(counts, what, bound, base):
        """Uniform positions among each table's `bound` resident keys, table by table."""
        of = torch.from_numpy(np.repeat(np.arange(T), counts)).to(DEVICE)
        u = torch.rand(int(counts.sum()), generator=_gen(seed, what), dtype=torch.float64, device=DEVICE)
        b = torch.from_numpy(np.asarray(bound)).to(DEVICE)[of]
        return torch.from_numpy(np.asarray(base)).to(DEVICE)[of] + (u * b).to(torch.int64)

    qpos = per_table(nq, 63, fill, start[:-1])
    miss = torch.rand(tot_q, generator=_gen(seed, 64), device=DEVICE) < 0.5
    q = _at(seed, torch.where(miss, qpos + (1 << 40), qpos))
    uk = _at(seed, per_table(nu, 65, fill, start[:-1]))
    uv = _index(seed, 66, tot_u, ADD_MAX) + 1
    wpos = np.repeat(start[:-1] + fill, win) + np.arange(tot_w) - np.repeat(np.cumsum(win) - win, win)
    wk = _at(seed, torch.from_numpy(wpos).to(DEVICE))
    wv = _values(wk)
    u64 = lambda n: torch.zeros(n, dtype=torch.int64, device=DEVICE)  # noqa: E731
    u8 = lambda n: torch.zeros(n, dtype=torch.uint8, device=DEVICE)  # noqa: E731
    out = {"insert": u8(tot_w), "upsert": u8(tot_u), "values": u64(tot_q), "status": u8(tot_q),
           "erased": u64(tot_w), "erase_status": u8(tot_w)}
    tables = [_table(c, int(s)) for s in caps]
    resident = _keys(seed, 0, int(start[-1]))
    items, setup = [], []
    iq = iu = iw = 0
    for i, t in enumerate(tables):
        a, b = int(start[i]), int(start[i] + fill[i])
        k = resident[a:b]
        setup.append((t, ws.BK_INSERT, k, _values(k), None, None, 0))
        Q, U, V = slice(iq, iq + int(nq[i])), slice(iu, iu + int(nu[i])), slice(iw, iw + int(win[i]))
        iq, iu, iw = Q.stop, U.stop, V.stop
        items += [(t, ws.BK_INSERT, wk[V], wv[V], None, out["insert"][V], 0),
                  (t, ws.BK_UPSERT, uk[U], uv[U], None, out["upsert"][U], 1, "add"),
                  (t, ws.BK_QUERY, q[Q], None, out["values"][Q], out["status"][Q], 2),
                  (t, ws.BK_ERASE, wk[V], None, out["erased"][V], out["erase_status"][V], 3)]
    first = ws.BatchPlan(setup)
    first.launch()
    first.close()
    return {"case": c, "tables": tables, "plan": ws.BatchPlan(items), "out": out}


def _prepare_serve(c, seed):
    T, R = c["tables"], c["requests"]
    caps = 1 << np.floor(np.log2(_sizes(c, 71, T, 1 << c["log2_min"], 1 << c["log2_max"]))).astype(np.int64)
    pairs = max(1, R // 2)
    table_of = np.random.RandomState(c["sizes"] * 31 + 72).randint(0, T, pairs)
    n_of = _sizes(c, 73, pairs, 16, c["ops_max"])
    server = ws.Server()
    ids = [server.add_table(int(s), c["scheme"], c["meta"]) for s in caps]
    total = int(2 * n_of.sum())
    pin = lambda dt: torch.empty(total, dtype=dt, pin_memory=True)  # noqa: E731
    ops, keys, vals, vo, st = pin(torch.uint8), pin(torch.int64), pin(torch.int64), pin(torch.int64), pin(torch.uint8)
    reqs, fills, at = [], [], 0
    for j in range(pairs):
        n, ti = int(n_of[j]), int(table_of[j])
        present = max(1, int(0.35 * caps[ti]) // int((table_of == ti).sum()))
        # each pair of requests has window keys of its own, disjoint from the resident ones
        sub = seed * 4099 + j + 1
        pair, m = _mixed_pair(sub, n, present, int(caps[ti]) // 50, 0.99)
        fills.append((ti, sub, present, m))
        for o, k, v in pair:
            a, b = at, at + n
            at = b
            ops[a:b], keys[a:b], vals[a:b] = o.cpu(), k.cpu(), v.cpu()
            reqs.append((ids[ti], a, b))
    h = {k: v.numpy() for k, v in (("ops", ops), ("keys", keys), ("vals", vals), ("vo", vo), ("st", st))}
    h["keys"], h["vals"], h["vo"] = (h[k].view(np.uint64) for k in ("keys", "vals", "vo"))
    # fill the tables through the server: the resident keys a request names, and the window keys it erases first
    for ti, sub, present, m in fills:
        k = torch.cat([_keys(sub, 0, present), _keys(sub, present + m, m)]).cpu().numpy()
        code = np.full(k.size, ws.MX_INSERT, np.uint8)
        for a in range(0, k.size, 1 << 22):
            server.submit(ids[ti], code[a:a + (1 << 22)], k[a:a + (1 << 22)], k[a:a + (1 << 22)] * np.int64(3))
        server.drain()
    return {"case": c, "server": server, "reqs": reqs, "h": h, "pinned": (ops, keys, vals, vo, st)}


def _run_serve(state):
    server, h = state["server"], state["h"]
    for tid, a, b in state["reqs"]:
        server.submit(tid, h["ops"][a:b], h["keys"][a:b], h["vals"][a:b], vals_out=h["vo"][a:b],
                      status_out=h["st"][a:b])
    server.drain()
    return {"values": h["vo"].view(np.int64), "status": h["st"]}


# ---------------------------------------------------------------------------
# work and expected results
# ---------------------------------------------------------------------------
def work(case):
    """Bytes no implementation avoids: keys, values and op codes read, results written, one 16-byte slot read per
    operation and written per change, a cleared table's slots written.  No floating-point work."""
    c = case
    query, upsert, insert, erase = 8 + 8 + 1 + 16, 16 + 1 + 32, 16 + 1 + 16, 8 + 9 + 32
    if c["kind"] == "lookup":
        b = c["n"] * query
    elif c["kind"] == "step":
        _, w = _counts(c)
        b = c["n"] * (2 * query + upsert) + w * (insert + erase)
    elif c["kind"] == "build":
        p, _ = _counts(c)
        b = 16 * _slots(c) + p * insert + max(1, int(c["probe"] * p)) * query
    elif c["kind"] == "groupby":
        p, _ = _counts(c)
        b = 16 * _slots(c) + c["n"] * 16 + p * (32 + query)
    elif c["kind"] == "mixed":
        b = 2 * c["n"] * (17 + 9 + 16 + 8)
    else:
        top = c["ops_max"]
        mean = (top - 256) / math.log(top / 256.0) if c["kind"] == "batched" else (top - 16) / math.log(top / 16.0)
        b = (c["tables"] if c["kind"] == "batched" else c["requests"]) * mean * 40
    return {"bytes": float(b), "flops": 0.0}


def exact(case, seed):
    """What run() returns on a new state, from the definition of a map (FOUND 1, INSERTED 2, MISS 0)."""
    c = case
    if c["kind"] not in ("lookup", "step", "build", "groupby"):
        return None
    p, w = _counts(c)
    d = _inputs(c, seed)
    u8 = lambda n, v: torch.full((n,), v, dtype=torch.uint8, device=DEVICE)  # noqa: E731
    if c["kind"] in ("lookup", "build"):
        v = torch.where(d["miss"], torch.zeros_like(d["q"]), _values(d["q"]))
        out = {"values": v, "status": (~d["miss"]).to(torch.uint8)}
        return out if c["kind"] == "lookup" else {"insert": u8(p, 2), **out}
    if c["kind"] == "groupby":
        sums = torch.zeros(p, dtype=torch.int64, device=DEVICE).index_add_(0, d["gi"], d["v"])
        seen = torch.zeros(p, dtype=torch.uint8, device=DEVICE)
        seen[d["gi"]] = 1
        return {"sums": sums, "status": seen}
    n = c["n"]
    add = torch.zeros(p, dtype=torch.int64, device=DEVICE).index_add_(0, d["ui"], d["uv"])
    return {"insert": u8(w, 2), "upsert": u8(n, 1), "present": _values(d["qk"]) + add[d["qi"]],
            "absent": torch.zeros(n, dtype=torch.int64, device=DEVICE), "absent_status": u8(n, 0),
            "erased": _values(d["wk"]), "erase_status": u8(w, 1)}
