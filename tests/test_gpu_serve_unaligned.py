"""A server request whose u64 arrays are page-locked but not 8-byte aligned (a
packed message: op bytes first, keys after them) is copied, not read in place,
and served like any other.  Needs a GPU."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _at(buf, off, a):
    """A copy of array a at byte `off` of the page-locked buffer."""
    v = buf[off: off + a.nbytes].view(a.dtype)
    v[:] = a
    return v


@pytest.mark.parametrize("shifts", [(0, 0, 0), (1, 0, 0), (0, 4, 0), (0, 0, 7), (3, 3, 3)])
@pytest.mark.parametrize("n", [1, 257, 5001])
def test_unaligned_request_is_copied(oracle_mod, n, shifts):
    import torch
    import paper_2509_16407_gb300 as ws
    from paper_2509_16407_gb300 import _lib
    ops, keys, vals = W.mixed_request_codes(8100 + n, n, 2500, 3)
    t = torch.empty(26 * n + 128, dtype=torch.uint8, pin_memory=True)
    buf = t.numpy()
    at = [32, 32 + 8 * (n + 2), 32 + 16 * (n + 2)]  # keys, values, results
    assert t.data_ptr() % 8 == 0
    k = _at(buf, at[0] + shifts[0], keys)
    v = _at(buf, at[1] + shifts[1], vals)
    vo = _at(buf, at[2] + shifts[2], np.full(n, 99, np.uint64))
    o = _at(buf, 32 + 24 * (n + 2), ops)
    st = _at(buf, 32 + 24 * (n + 2) + n, np.full(n, 99, np.uint8))
    req = _lib.WsRequest(0, 0, o.ctypes.data, k.ctypes.data, v.ctypes.data, vo.ctypes.data, st.ctypes.data, n, 0)
    in_place = ws.lib().ws_debug_request_in_place(ctypes.byref(req))
    assert in_place == (1 if shifts == (0, 0, 0) else 0)  # before anything is launched
    om = oracle_mod.OracleMap()
    ov, os_ = om.mixed(ops, keys, vals)
    sv = ws.Server()
    tid = sv.add_table(1 << 13, "double", False)
    sv.submit(tid, o, k, v, vals_out=vo, status_out=st)
    done = sv.drain()
    assert len(done) == 1 and done[0]["status"] == 0
    q = ops == W.MX_QUERY
    assert (vo[q] == ov[q]).all() and (st[q] == os_[q]).all()
    for code in np.unique(ops):  # the copies of one key race: as many of each status
        m = ops == code
        assert (np.bincount(st[m], minlength=6) == np.bincount(os_[m], minlength=6)).all()
    assert sv.count(tid) == om.count()
    sv.close()
