"""Server requests in page-locked buffers, which the kernel's blocks copy
themselves: odd sizes, slices that start at any byte, missing values and
results, chunk edges, and page-locked requests between pageable ones give the
results of the oracle's replay.  Needs a GPU."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [1, 31, 255, 256, 257, 2047, 2048, 2049, 4097, 7001]


@pytest.mark.parametrize("pinned", ["all", "alternate", "but_status"])
@pytest.mark.parametrize("scheme,meta,tile", [("double", False, 8), ("double", True, 4), ("p2", False, 8),
                                               ("p2", True, 4), ("double", False, 16)])
def test_pinned_requests(oracle_mod, scheme, meta, tile, pinned):
    import torch
    import paper_2509_16407_gb300 as ws
    sv = ws.Server()
    tid = sv.add_table(1 << 13, scheme, meta, tile)
    om = oracle_mod.OracleMap()
    keep, want = [], []

    def buf(a, pin, odd):
        """A copy of array a that starts `odd` elements into its allocation."""
        t = torch.empty(a.nbytes + 64, dtype=torch.uint8, pin_memory=pin)
        keep.append(t)
        v = t.numpy()[odd * a.itemsize: odd * a.itemsize + a.nbytes].view(a.dtype)
        v[:] = a
        return v

    reqs = []
    for i, n in enumerate(SIZES):
        ops, keys, vals = W.mixed_request_codes(7000 + i, n, 2500, 3)
        pin = pinned != "alternate" or i % 2 == 0
        no_vals = i % 4 == 3
        if no_vals:
            ops = np.where((ops == W.MX_QUERY) | (ops == W.MX_ERASE), ops, W.MX_ADD).astype(np.uint8)
        ov, os_ = om.mixed(ops, keys, np.zeros_like(vals) if no_vals else vals)
        vo = buf(np.zeros(n, np.uint64), pin, i % 3)
        st = buf(np.full(n, 99, np.uint8), pin and pinned != "but_status", i % 7)
        reqs.append((buf(ops, pin, i % 5), buf(keys, pin, i % 4), None if no_vals else buf(vals, pin, i % 2),
                     vo if i % 5 != 4 else None, st))
        want.append((ops, keys, ov, os_))
    for ops, keys, vals, vo, st in reqs:
        sv.submit(tid, ops, keys, vals, want_values=vo is not None, vals_out=vo, status_out=st)
    done = sv.drain()
    assert len(done) == len(reqs) and all(c["status"] == 0 for c in done)
    for (ops, keys, ov, os_), (_, _, _, vo, st) in zip(want, reqs):
        q = ops == W.MX_QUERY
        assert (st[q] == os_[q]).all()
        for code in np.unique(ops):  # the copies of one key race: as many of each status
            m = ops == code
            assert (np.bincount(st[m], minlength=6) == np.bincount(os_[m], minlength=6)).all()
        if vo is not None:
            assert (vo[q] == ov[q]).all()
    assert sv.count(tid) == om.count()
    sv.close()
