"""Inserts whose inserters meet: tables built from nothing by one call, several
ops in flight per bucket and per lock bit, with and without copies of a key.
Exactly one copy of a key reports INSERTED, the map equals the oracle's and
the layout rules hold (EMPTY slots a suffix, no duplicate, two-choice and
iceberg early exits).  Needs a GPU."""
import numpy as np
import pytest

import workloads as W
from tests._gpu import DESIGNS, DESIGN_IDS, check_layout, dev, host

pytestmark = pytest.mark.gpu

CASES = [(s, m, 0) for s, m in DESIGNS] + [("p2", False, 16), ("p2", False, 8), ("double", False, 32)]
CASE_IDS = DESIGN_IDS + ["P2HT-B16", "P2HT-B8", "DoubleHT-B32"]


@pytest.fixture(scope="module")
def ws():
    import torch
    assert torch.cuda.is_available()
    from paper_2509_16407_gb300 import build as b
    b.build()
    import paper_2509_16407_gb300 as ws
    ws.lib()
    return ws


@pytest.mark.parametrize("op", ["insert", "add", "replace"])
@pytest.mark.parametrize("copies", [1, 3])
@pytest.mark.parametrize("log2", [7, 11, 16])
@pytest.mark.parametrize("scheme,meta,B", CASES, ids=CASE_IDS)
def test_build_from_nothing(ws, oracle_mod, scheme, meta, B, log2, copies, op):
    t = ws.Table(1 << log2, scheme, meta, bucket_slots=B)
    n = int((0.35 if B == 8 else 0.55) * (1 << log2))  # no insert may fail, whatever the interleaving
    uniq = W.distinct_keys(4200 + log2, n)
    keys = np.repeat(uniq, copies)[W.permutation(4300 + log2, n * copies)]
    vals = W.mix13(keys) | np.uint64(1)  # one value per key: which copy wins does not show
    got = host(t.upsert(dev(keys), dev(vals), op=op, return_status=True))
    assert set(np.unique(got)) <= {ws.INSERTED, ws.FOUND}
    assert (got == ws.INSERTED).sum() == n
    first = np.unique(keys[got == ws.INSERTED])
    assert first.size == n  # one INSERTED copy per key
    with np.errstate(over="ignore"):
        want = (W.mix13(uniq) | np.uint64(1)) * np.uint64(copies if op == "add" else 1)
    v, st = t.query(dev(uniq), return_status=True)
    assert (host(st) == ws.FOUND).all() and (host(v) == want).all()
    check_layout(oracle_mod, t, n)
    # the same keys after an erase: freed slots are claimed again
    ev, es = t.erase(dev(uniq[::2]), return_values=True, return_status=True)
    assert (host(es) == ws.FOUND).all() and (host(ev) == want[::2]).all()
    again = host(t.upsert(dev(keys), dev(vals), op=op, return_status=True))
    assert (again == ws.INSERTED).sum() == uniq[::2].size
    assert t.count() == n
    check_layout(oracle_mod, t, n)
    assert t.last_error()["status"] == 0
    t.close()


@pytest.mark.parametrize("slices", [2, 9])
@pytest.mark.parametrize("log2", [12, 17])
@pytest.mark.parametrize("scheme,meta,B", [c for c in CASES if c[0] != "double"],
                         ids=[i for i, c in zip(CASE_IDS, CASES) if c[0] != "double"])
def test_fill_across_the_lock_line(ws, oracle_mod, scheme, meta, B, log2, slices):
    """Filled to 0.8 in slices, so that calls insert lock-free, lock first and
    on either side of the load where that changes; every key twice per call.
    8-slot buckets may report FULL at 0.6 (a few of 10^6 keys, whatever the
    order): then both of the key's buckets must be full."""
    t = ws.Table(1 << log2, scheme, meta, bucket_slots=B)
    n = int((0.6 if B == 8 else 0.8) * (1 << log2))
    uniq = W.distinct_keys(4400 + log2, n)
    om = oracle_mod.OracleMap()
    failed = []
    for i in range(slices):
        part = uniq[i * n // slices:(i + 1) * n // slices]
        keys = np.concatenate([part, part])[W.permutation(4500 + i, 2 * part.size)]
        vals = W.mix13(keys)
        st = host(t.insert(dev(keys), dev(vals), return_status=True))
        bad = np.unique(keys[st == ws.FAIL_FULL])
        failed.append(bad)
        ok = part.size - bad.size
        om.insert(keys[~np.isin(keys, bad)], vals[~np.isin(keys, bad)])
        assert (st == ws.INSERTED).sum() == ok and (st == ws.FOUND).sum() == ok
        assert (st == ws.FAIL_FULL).sum() == 2 * bad.size
        assert np.unique(keys[st == ws.INSERTED]).size == ok
    failed = np.concatenate(failed)
    assert failed.size <= (1e-4 * n if B == 8 else 0)
    assert t.count() == n - failed.size == om.count()
    v, st = t.query(dev(uniq), return_status=True)
    want, wst = om.query(uniq)
    assert (host(v) == want).all() and (host(st) == wst).all()
    _, L = check_layout(oracle_mod, t, n - failed.size)
    if failed.size:
        assert oracle_mod.candidates_full(L["slots"], L["tags"], L["nb"], L["B"], L["scheme"], L["pmax"], L["seed1"],
                                          L["seed2"], failed).all()
    t.close()


@pytest.mark.parametrize("meta", [False, True], ids=["P2HT", "P2HT(M)"])
@pytest.mark.parametrize("kind", ["insert", "add"])
def test_batched_fill_counts_as_load(ws, meta, kind):
    """A two-choice table that a batch plan has filled to 0.7 is no low-load
    table to the next single-table insert: every key takes its lock (shown by
    locks that are all taken), as in a table filled by single-table calls."""
    S = 1 << 14
    t = ws.Table(S, "p2", meta, tile=8, spin_limit=64)
    n = int(0.7 * S)
    keys = W.distinct_keys(4600, n + 1000)
    kd, st = dev(keys[:n]), dev(np.zeros(n, np.uint8))
    item = (t, ws.BK_INSERT if kind == "insert" else ws.BK_UPSERT, kd, kd, None, st, 0)
    plan = ws.BatchPlan([item + (("add",) if kind == "add" else ())])
    assert plan.info()["fallback_items"] == 0
    plan.launch()
    assert (host(st) == ws.INSERTED).all() and t.count() == n
    t.debug_fill_locks(True)
    new = dev(keys[n:])
    assert (host(t.insert(new, new, return_status=True)) == ws.FAIL_TIMEOUT).all()
    t.debug_fill_locks(False)
    assert (host(t.insert(new, new, return_status=True)) == ws.INSERTED).all()
    plan.close()
    t.close()


@pytest.mark.parametrize("scheme,plain", [("iceberg", False), ("p2", True)])
def test_served_fill_counts_as_load(ws, scheme, plain):
    """The same for a table that a server's requests have filled to 0.8 by
    single-table kernels (no menu entry, or one launch per request)."""
    import ctypes
    S = 1 << 14
    sv = ws.Server(grow_at=0, plain=plain)
    tid = sv.add_table(S, scheme, True)
    n = int(0.8 * S)
    keys = W.distinct_keys(4700, n + 500)
    sv.submit(tid, np.full(n, ws.MX_INSERT, np.uint8), keys[:n], keys[:n])
    done = sv.drain()
    assert len(done) == 1 and (done[0]["st"] == ws.INSERTED).all()
    h, L = sv.table_handle(tid), ws.lib()
    st = np.zeros(500, np.uint8)
    new = np.ascontiguousarray(keys[n:])
    for locked, want in ((1, ws.FAIL_TIMEOUT), (0, ws.INSERTED)):
        assert L.ws_set_spin_limit(h, 64 if locked else 65536) == 0 and L.ws_debug_fill_locks(h, locked, None) == 0
        assert L.ws_insert_ex(h, new.ctypes.data, new.ctypes.data, 500, st.ctypes.data, None) in (0, 5)
        assert sv.count(tid) == n + (0 if locked else 500)  # waits for the call
        assert (st == want).all()
    sv.close()
