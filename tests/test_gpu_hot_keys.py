"""Upserts of a few very frequent keys, which a block settles in shared memory
once it knows them: one INSERTED copy per key, exact sums and maxima, one of
the given values under replace, and a map equal to the oracle's.  Needs a GPU."""
import numpy as np
import pytest

import workloads as W
from tests._gpu import DESIGNS, DESIGN_IDS, check_layout, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["add", "max", "replace", "insert"])
@pytest.mark.parametrize("n_keys", [1, 5, 70, 4000])  # below and above what a block keeps (64)
@pytest.mark.parametrize("scheme,meta", DESIGNS, ids=DESIGN_IDS)
def test_frequent_keys(oracle_mod, scheme, meta, n_keys, op):
    import torch
    import paper_2509_16407_gb300 as ws
    n = 300007
    t = ws.Table(1 << 14, scheme, meta)
    uniq = W.distinct_keys(600 + n_keys, n_keys)
    old = uniq[::2]  # half of the keys are there before
    with np.errstate(over="ignore"):
        t.insert(dev(old), dev(old * np.uint64(7)))
    pick = (W.zipf(601, n, n_keys, 1.05) - 1) if n_keys > 1 else np.zeros(n, np.int64)
    keys = uniq[pick]
    vals = W.splitmix64(602, n) >> np.uint64(1)
    st = host(t.upsert(dev(keys), dev(vals), op=op, return_status=True))
    here = np.unique(pick)
    new = here[here % 2 == 1]
    assert (st == ws.INSERTED).sum() == new.size and (st == ws.FOUND).sum() == n - new.size
    assert np.unique(keys[st == ws.INSERTED]).size == new.size
    base = np.zeros(n_keys, np.uint64)
    with np.errstate(over="ignore"):
        base[::2] = old * np.uint64(7)
    v, f = t.query(dev(uniq), return_status=True)
    v, f = host(v), host(f)
    present = np.zeros(n_keys, bool)
    present[::2] = True
    present[here] = True
    assert (f == np.where(present, ws.FOUND, ws.MISS)).all()
    if op == "add":
        want = base.copy()
        np.add.at(want, pick, vals)
        assert (v == want).all()
    elif op == "max":
        want = base.copy()
        np.maximum.at(want, pick, vals)
        assert (v == want).all()
    else:
        given = set(zip(pick.tolist(), vals.tolist()))
        seen = np.zeros(n_keys, bool)
        seen[here] = True
        for i in range(n_keys):
            if not seen[i] or (op == "insert" and i % 2 == 0):
                assert v[i] == base[i]  # never named, or kept by insert-if-unique
            else:
                assert (i, int(v[i])) in given
    check_layout(oracle_mod, t, int(present.sum()))
    assert t.last_error()["status"] == 0
    # page-locked inputs, no statuses
    if op == "add":
        hk, hv = (torch.from_numpy(x.view(np.int64)).pin_memory() for x in (keys, vals))
        t.upsert(hk, hv, op="add")
        torch.cuda.synchronize()
        np.add.at(want, pick, vals)
        assert (host(t.query(dev(uniq))) == want).all()
    t.close()


@pytest.mark.parametrize("n_keys", [12, 400])
@pytest.mark.parametrize("scheme,meta", DESIGNS, ids=DESIGN_IDS)
def test_frequent_keys_in_mixed_batches(oracle_mod, scheme, meta, n_keys):
    """Every code on its own skewed keys, the added ones above all: sums,
    maxima, queried values and the counts of each status are the oracle's."""
    import paper_2509_16407_gb300 as ws
    n = 400003
    t = ws.Table(1 << 14, scheme, meta)
    om = oracle_mod.OracleMap()
    uniq = W.distinct_keys(800 + n_keys, 6 * n_keys)
    old = uniq[::2]
    t.insert(dev(old), dev(old))
    om.insert(old, old)
    code = np.where(W.splitmix64(801, n) % np.uint64(3) == 0, W.splitmix64(802, n) % np.uint64(6), W.MX_ADD).astype(np.uint8)
    keys = uniq.reshape(6, n_keys)[code, W.zipf(803, n, n_keys, 1.05) - 1]  # a key has one code
    vals = W.splitmix64(804, n) >> np.uint64(8)
    one = (code == W.MX_REPLACE) | (code == W.MX_INSERT)
    vals[one] = W.mix13(keys[one])  # which copy wins does not show
    v, st = t.mixed(dev(code), dev(keys), dev(vals))
    wv, wst = om.mixed(code, keys, vals)
    v, st = host(v), host(st)
    for c in range(6):
        m = code == c
        assert (np.bincount(st[m], minlength=6) == np.bincount(wst[m], minlength=6)).all()
        if c == W.MX_QUERY:
            assert (v[m] == wv[m]).all()
        elif c != W.MX_ERASE:
            assert (v[m] == 0).all()
    got, gst = t.query(dev(uniq), return_status=True)
    want, ost = om.query(uniq)
    assert (host(got) == want).all() and (host(gst) == ost).all()
    assert t.count() == om.count()
    check_layout(oracle_mod, t, om.count())
    t.close()
