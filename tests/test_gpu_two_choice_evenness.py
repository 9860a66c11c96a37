"""Two-choice tables of a few hundred buckets filled by one or two calls, every
key of a call in flight at once: concurrent placement leaves about as few keys
without a slot as placing the keys one after another does.  Needs a GPU."""
import numpy as np
import pytest

import workloads as W
from tests._gpu import dev

pytestmark = pytest.mark.gpu

LOG2, TABLES = 14, 24

CASES = [  # metadata, bucket slots, final load, how the table is filled
    (False, 32, 0.95, "insert"), (False, 32, 0.95, "add"), (False, 32, 0.95, "two_inserts"),
    (True, 32, 0.95, "insert"), (True, 32, 0.95, "add"), (True, 32, 0.95, "two_inserts"),
    (False, 16, 0.9, "insert"), (False, 16, 0.9, "add"),
    (False, 8, 0.9, "insert"), (False, 8, 0.9, "add"),
]


def placed_in_order(oracle, keys, nb, B, seed1, seed2):
    """Keys without a slot when they are placed one after another (b_0 while it
    is below 3/4, else the less loaded bucket, the other one when that is full)."""
    b0 = oracle.primary_bucket(keys, nb, seed1).astype(np.int64)
    b1 = oracle.primary_bucket(keys, nb, seed2).astype(np.int64)  # the second hash has its own seed
    b1 = np.where(b1 == b0, (b0 + 1) % nb, b1)
    occ, full = [0] * nb, 0
    for x, y in zip(b0.tolist(), b1.tolist()):
        c = x if occ[x] < B * 3 // 4 or occ[y] >= occ[x] else y
        if occ[c] == B:
            c = y if c == x else x
        if occ[c] == B:
            full += 1
        else:
            occ[c] += 1
    return full


@pytest.mark.parametrize("meta,B,load,how", CASES)
def test_keys_without_a_slot(oracle_mod, meta, B, load, how):
    import paper_2509_16407_gb300 as ws
    t = ws.Table(1 << LOG2, "p2", meta, bucket_slots=B)
    inf = t.info()
    n = int(load * inf["slots"])
    cuts = [0, int(0.55 * inf["slots"]), n] if how == "two_inserts" else [0, n]
    got = want = 0
    for s in range(TABLES):
        keys = W.distinct_keys(5200 + s, n)
        t.clear()
        for a, b in zip(cuts, cuts[1:]):
            d = dev(keys[a:b])
            t.upsert(d, d, op="add" if how == "add" else "insert")
        e = t.last_error()
        assert e["timeout"] == 0 and t.count() == n - e["full"]
        got += e["full"]
        want += placed_in_order(oracle_mod, keys, inf["buckets"], B, inf["seed1"], inf["seed2"])
    # A claim takes the emptier of the buckets as they are when it is made, so
    # only the order of the keys differs: a quarter more keys without a slot
    # than in the given order, and eight more per table (0.05% of its keys).
    assert got <= 1.25 * want + 8 * TABLES, (got / TABLES, want / TABLES)
    t.close()
