"""Skewed upserts and mixed batches on either side of the size from which a launch
looks for frequent keys (more than one op per lane of a full grid): sums, maxima
and counts of each status are the oracle's.  Needs a GPU."""
import numpy as np
import pytest

import workloads as W
from tests._gpu import DESIGNS, DESIGN_IDS, dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("over", [-1, 0, 1, 33, 12345])
@pytest.mark.parametrize("op", ["add", "max", "mixed"])
@pytest.mark.parametrize("scheme,meta", DESIGNS, ids=DESIGN_IDS)
def test_sizes_around_the_line(oracle_mod, scheme, meta, op, over):
    import torch
    import paper_2509_16407_gb300 as ws
    lanes = torch.cuda.get_device_properties(0).multi_processor_count * 4 * 256
    n = lanes + over
    t = ws.Table(1 << 14, scheme, meta)
    om = oracle_mod.OracleMap()
    uniq = W.distinct_keys(900, 2000)
    t.insert(dev(uniq[::2]), dev(uniq[::2]))
    om.insert(uniq[::2], uniq[::2])
    keys = uniq[W.zipf(901, n, 2000, 1.05) - 1]
    vals = W.splitmix64(902, n) >> np.uint64(1)
    if op == "mixed":
        code = np.where(W.mix13(keys) % np.uint64(3) == 0, W.MX_QUERY, W.MX_ADD).astype(np.uint8)
        v, st = t.mixed(dev(code), dev(keys), dev(vals))
        wv, wst = om.mixed(code, keys, vals)
        q = code == W.MX_QUERY
        assert (host(v)[q] == wv[q]).all()
    else:
        st = t.upsert(dev(keys), dev(vals), op=op, return_status=True)
        wst = om.upsert(keys, vals, ws.UPSERT_OPS[op])
    assert (np.bincount(host(st), minlength=6) == np.bincount(wst, minlength=6)).all()
    got, gst = t.query(dev(uniq), return_status=True)
    want, ost = om.query(uniq)
    assert (host(got) == want).all() and (host(gst) == ost).all()
    assert t.count() == om.count()
    t.close()
