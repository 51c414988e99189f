"""Prefill attention where one request's items are numbered head by head (its K
and V exceed 64 MB) and another's tile by tile, with the keys of an item whole and
split over a cluster: sampled rows of every tile against the float64 oracle, with
the suite's tolerance.  Items of a single step: the item slots change hands as
often as they can."""
import numpy as np
import pytest

import oracle
from paper_2505_23970_gb300 import binding as gcb
from paper_2505_23970_gb300 import workloads as wl
from paper_2505_23970_gb300.harness import DeviceBatch

from ._util import assert_attn_close, gather_rows, sample_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("new", [[700, 333], [40, 17]], ids=["whole", "split"])
def test_items_by_head_and_by_tile(new):
    w = wl.custom("by-head", 2, 16, 2, 128, 64, [66000, 500], new, seed=sum(new))
    assert (66000 + new[0]) * 2 > 131072 > (500 + new[1]) * 2
    db = DeviceBatch(w)
    db.run()
    assert db.check() == gcb.GC_OK
    pool = w.empty_pool()
    oracle.kv_restore(pool, w.host_src(), w.prefix_blocks())
    k, v = w.kv_new()
    oracle.kv_append(pool, 0, k, v, w.block_table, w.prefix_lens, w.cu_new_lens)
    rows = sample_rows(w, 256)
    ref = oracle.prefix_attn_rows(w.q(), pool, 0, w.block_table, w.prefix_lens, w.cu_new_lens,
                                  w.scale, rows)
    got = gather_rows(db.out_f64(), w, rows)
    assert_attn_close(got, ref, "by head")
    assert np.isfinite(db.out_f64()).all()
    db.close()


def test_items_of_one_step():
    """Five times as many items as pairs, one K/V step each, of 13 to 16 tokens
    (the last rows of a tile missing) behind 0 to 110 cached ones."""
    n = [13 + b % 4 for b in range(190)]
    P = [(7 * b) % 111 for b in range(190)]
    w = wl.custom("one-step", 190, 32, 2, 128, 16, P, n, seed=3)
    db = DeviceBatch(w)
    db.run()
    assert db.check() == gcb.GC_OK
    pool = w.empty_pool()
    oracle.kv_restore(pool, w.host_src(), w.prefix_blocks())
    k, v = w.kv_new()
    oracle.kv_append(pool, 0, k, v, w.block_table, w.prefix_lens, w.cu_new_lens)
    ref = oracle.prefix_attn(w.q(), pool, 0, w.block_table, w.prefix_lens, w.cu_new_lens, w.scale)
    assert_attn_close(db.out_f64(), ref, "one step")
    db.close()
