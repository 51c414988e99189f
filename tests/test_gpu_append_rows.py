"""gc_kv_append where a thread's words fall on different rows: tokens of fewer
words than a warp moves at once, head counts that are no power of two, requests
without new tokens, a call of a single token.  Bit for bit the oracle's pool."""
import numpy as np
import pytest

import oracle
from paper_2505_23970_gb300 import binding as gcb
from paper_2505_23970_gb300 import workloads as wl
from paper_2505_23970_gb300.harness import DeviceBatch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hkv,d,ps,P,n", [
    (1, 64, 16, [5, 0, 31, 16, 250], [1, 0, 33, 130, 7]),
    (3, 64, 32, [0, 100], [65, 3]),
    (5, 128, 16, [17, 0, 63], [1, 200, 15]),
    (8, 128, 128, [127, 1], [2, 1000]),
    (2, 128, 64, [700], [1]),
])
def test_append_rows(Hkv, d, ps, P, n):
    w = wl.custom("append-rows", len(P), Hkv, Hkv, d, ps, P, n, seed=Hkv + d)
    db = DeviceBatch(w)
    db.append()
    assert db.check() == gcb.GC_OK
    pool = w.empty_pool()
    k, v = w.kv_new()
    oracle.kv_append(pool, 0, k, v, w.block_table, w.prefix_lens, w.cu_new_lens)
    assert np.array_equal(db.pool_bits(), pool)
    db.close()
