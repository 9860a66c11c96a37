"""Which calls and server requests write their results in place, and that every
way gives the oracle's results: insert, upsert, erase and mixed calls with
page-locked results around the sizes where writing in place ends, and results
that lie inside other inputs or one byte off them.  Needs a GPU."""
import ctypes

import numpy as np
import pytest

import workloads as W
from tests._gpu import dev

pytestmark = pytest.mark.gpu

N_SLOTS = 1 << 20


class _Buf:
    """Page-locked memory with arrays at chosen byte offsets (8-byte aligned base)."""

    def __init__(self, size):
        import torch
        self.t = torch.empty(size, dtype=torch.uint8, pin_memory=True)
        self.a = self.t.numpy()
        self.base = self.t.data_ptr()
        assert self.base % 8 == 0

    def put(self, off, arr):
        v = self.a[off: off + arr.nbytes].view(arr.dtype)
        v[:] = arr
        return v


def _counts_equal(ops, got, want):
    for code in np.unique(ops):  # the copies of one key race: as many of each status
        m = ops == code
        assert (np.bincount(got[m], minlength=6) == np.bincount(want[m], minlength=6)).all(), code


@pytest.mark.parametrize("n", [1, 257, (1 << 18) - 1, 1 << 18, (1 << 18) + 1, (1 << 19) - 1, 1 << 19, (1 << 19) + 1])
@pytest.mark.parametrize("scheme,meta", [("double", False), ("p2", True)])
def test_results_of_every_call(oracle_mod, scheme, meta, n):
    import torch
    import paper_2509_16407_gb300 as ws
    t = ws.Table(N_SLOTS, scheme, meta)
    om = oracle_mod.OracleMap()
    pin = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int64 if a.dtype == np.uint64 else a.dtype)).pin_memory()
    keys = W.distinct_keys(91, n)
    vals = W.splitmix64(92, n)
    st = t.insert(pin(keys), pin(vals), return_status=True)
    assert st.is_pinned()
    torch.cuda.synchronize()
    assert (st.numpy() == om.insert(keys, vals)).all()
    st = t.upsert(pin(keys), pin(vals), op="add", return_status=True)
    torch.cuda.synchronize()
    assert (st.numpy() == om.upsert(keys, vals, 0)).all()
    ops, mk, mv = W.mixed_batch_codes(93, n_ops=n, universe=max(4, n // 3), universe_seed=7)
    vo, st = t.mixed(torch.from_numpy(ops).pin_memory(), pin(mk), pin(mv))
    torch.cuda.synchronize()
    ov, os_ = om.mixed(ops, mk, mv)
    q = ops == W.MX_QUERY
    assert (vo.numpy().view(np.uint64)[q] == ov[q]).all() and (st.numpy()[q] == os_[q]).all()
    _counts_equal(ops, st.numpy(), os_)
    ev, st = t.erase(pin(keys), return_values=True, return_status=True)
    torch.cuda.synchronize()
    wv, ws_ = om.erase(keys)
    assert (ev.numpy().view(np.uint64) == wv).all() and (st.numpy() == ws_).all()
    assert t.count() == om.count()
    t.close()


# Where the results of a mixed batch of n ops lie: (values, status), as byte
# offsets from (name of an array, offset in it).  None: memory of their own.
PLACES = {
    "apart": (None, None),
    "values_over_keys": (("keys", 0), None),
    "values_over_values": (("vals", 0), None),
    "values_one_off_keys": (("keys", -8), None),
    "values_one_off_values": (("vals", 8), None),
    "values_over_ops": (("ops", 0), None),
    "status_over_ops": (None, ("ops", 0)),
    "status_one_off_ops": (None, ("ops", 1)),
    "status_in_keys": (None, ("keys", 8)),
    "status_in_values": (None, ("vals", 3)),
}
IN_PLACE = {"apart", "values_over_keys", "values_over_values", "status_over_ops"}


def _place(place, ops, keys, vals):
    n = keys.size
    gap = 64
    at, off = {}, gap
    for name, size in (("keys", 8 * n), ("vals", 8 * n), ("ops", 9 * n), ("vo", 8 * n), ("st", n)):
        at[name] = (off + 7) // 8 * 8
        off = at[name] + size + gap
    b = _Buf(off + gap)
    k, v, o = b.put(at["keys"], keys), b.put(at["vals"], vals), b.put(at["ops"], ops)
    pv, ps = PLACES[place]
    vo_at = at["vo"] if pv is None else at[pv[0]] + pv[1]
    st_at = at["st"] if ps is None else at[ps[0]] + ps[1]
    return b, k, v, o, b.a[vo_at: vo_at + 8 * n].view(np.uint64), b.a[st_at: st_at + n]


@pytest.mark.parametrize("place", sorted(PLACES))
@pytest.mark.parametrize("n", [33, 6001])
def test_results_that_overlap_inputs(oracle_mod, place, n):
    import torch
    import paper_2509_16407_gb300 as ws
    from paper_2509_16407_gb300 import _lib
    ops, keys, vals = W.mixed_request_codes(9400 + n, n, 2500, 5)
    om = oracle_mod.OracleMap()
    ov, os_ = om.mixed(ops, keys, vals)
    q = ops == W.MX_QUERY
    L = ws.lib()

    b, k, v, o, vo, st = _place(place, ops, keys, vals)
    t = ws.Table(1 << 13)
    assert L.ws_mixed(t.handle, o.ctypes.data, k.ctypes.data, v.ctypes.data, vo.ctypes.data, st.ctypes.data, n,
                      t._stream(None)) == 0
    torch.cuda.synchronize()
    assert (vo[q] == ov[q]).all()
    _counts_equal(ops, st, os_)
    assert t.count() == om.count()
    t.close()

    b, k, v, o, vo, st = _place(place, ops, keys, vals)
    req = _lib.WsRequest(0, 0, o.ctypes.data, k.ctypes.data, v.ctypes.data, vo.ctypes.data, st.ctypes.data, n, 0)
    assert L.ws_debug_request_in_place(ctypes.byref(req)) == (place in IN_PLACE)
    sv = ws.Server()
    tid = sv.add_table(1 << 13)
    sv.submit(tid, o, k, v, vals_out=vo, status_out=st)
    done = sv.drain()
    assert len(done) == 1 and done[0]["status"] == 0
    assert (vo[q] == ov[q]).all()
    _counts_equal(ops, st, os_)
    assert sv.count(tid) == om.count()
    sv.close()
