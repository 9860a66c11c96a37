"""Small calls with page-locked buffers write their results in place: odd
sizes on either side of where that ends, results over the keys themselves,
and results that overlap other inputs.  Needs a GPU."""
import numpy as np
import pytest

import workloads as W
from tests._gpu import dev

pytestmark = pytest.mark.gpu


def _pinned(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int64 if a.dtype == np.uint64 else a.dtype)).pin_memory()


@pytest.mark.parametrize("n", [1, 33, 100003, (1 << 19) - 1, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("scheme,meta", [("double", False), ("p2", False), ("iceberg", True)])
def test_results_in_place(oracle_mod, scheme, meta, n):
    import torch
    import paper_2509_16407_gb300 as ws
    t = ws.Table(1 << 16, scheme, meta)
    om = oracle_mod.OracleMap()
    keys = W.distinct_keys(31, 30000)
    vals = W.splitmix64(32, keys.size)
    t.insert(dev(keys), dev(vals))
    om.insert(keys, vals)
    q = W.distinct_keys(31, 60000)[W.splitmix64(33, n) % np.uint64(60000)]
    want, wst = om.query(q)
    v, st = t.query(_pinned(q), return_status=True)
    torch.cuda.synchronize()
    assert (v.numpy().view(np.uint64) == want).all() and (st.numpy() == wst).all()
    over = _pinned(q)  # results over the keys
    t.query(over, out=over)
    torch.cuda.synchronize()
    assert (over.numpy().view(np.uint64) == want).all()
    both = _pinned(np.concatenate([np.zeros(1, np.uint64), q]))  # results one element before the keys
    t.query(both[1:], out=both[:n])
    torch.cuda.synchronize()
    assert (both.numpy().view(np.uint64)[:n] == want).all()
    ev, es = t.erase(_pinned(keys[: min(n, 5000)]), return_values=True, return_status=True)
    torch.cuda.synchronize()
    assert (ev.numpy().view(np.uint64) == vals[: ev.numel()]).all() and (es.numpy() == ws.FOUND).all()
    t.close()
