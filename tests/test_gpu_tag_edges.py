"""Fingerprints at the edges of the word-parallel tag scans: keys that differ
only above their low 16 bits, with tags next to the reserved values, to the
sign bit of a 16-bit field and to each other, so that buckets hold many equal
and nearly equal tags.  Needs a GPU."""
import numpy as np
import pytest

import workloads as W
from tests._gpu import check_layout, dev, host

pytestmark = pytest.mark.gpu

TAGS = np.array([0, 1, 2, 3, 0x7ffe, 0x7fff, 0x8000, 0x8001, 0xfffe, 0xffff], np.uint64)


@pytest.mark.parametrize("scheme", ["double", "p2", "iceberg"])
@pytest.mark.parametrize("n_tags", [1, 3, 10])
def test_equal_and_neighbouring_tags(oracle_mod, scheme, n_tags):
    import paper_2509_16407_gb300 as ws
    for shift in range(0, TAGS.size, n_tags):
        tags = np.roll(TAGS, -shift)[:n_tags]
        hi = (W.splitmix64(91 + shift, 1200) >> np.uint64(17)) + np.uint64(1)
        keys = np.unique((hi << np.uint64(16)) | tags[np.arange(hi.size) % n_tags])
        keys = keys[W.permutation(92, keys.size)]
        present, absent = keys[:600], keys[600:]
        t = ws.Table(1 << 10, scheme, True)
        om = oracle_mod.OracleMap()
        vals = W.mix13(present)
        assert (host(t.insert(dev(present), dev(vals), return_status=True)) == om.insert(present, vals)).all()
        for q in (present, absent):
            v, st = t.query(dev(q), return_status=True)
            want, wst = om.query(q)
            assert (host(v) == want).all() and (host(st) == wst).all()
        ev, es = t.erase(dev(keys[::3]), return_values=True, return_status=True)
        wv, wes = om.erase(keys[::3])
        assert (host(ev) == wv).all() and (host(es) == wes).all()
        both = np.concatenate([present, absent[:100]])
        assert (host(t.upsert(dev(both), dev(both), op="add", return_status=True)) == om.upsert(both, both, 0)).all()
        v, st = t.query(dev(keys), return_status=True)
        want, wst = om.query(keys)
        assert (host(v) == want).all() and (host(st) == wst).all()
        check_layout(oracle_mod, t, om.count())
        t.close()
