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
from paper_2505_23970_gb300.harness import DeviceBatch, _i32, bf16_tensor

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


@pytest.mark.parametrize("d,G,P,windows", [
    (64, 16, 200, [(0, 100), (50, 100)]),
    (128, 16, 200, [(0, 100), (50, 100)]),
    (128, 16, 5000, [(0, 32), (8, 32), (16, 32)]),
    (128, 4, 3000, [(0, 128), (16, 128), (32, 128)]),
], ids=["d64", "whole", "split in 4", "split in 4, fewer heads"])
def test_requests_that_share_rows(d, G, P, windows):
    """Requests over overlapping windows (first row, rows) of one sequence's new
    tokens: new_lens sums up to more than the rows there are, and the items to more
    than a grid sized by the rows.  Every row is written, by each request alike."""
    import torch
    ps, Hkv, T = 16, 2, max(a + n for a, n in windows)
    pages = -(-(P + T) // ps)
    pool = wl.normal_bf16(11, 1, (1, 2, pages, Hkv, ps, d))
    q = wl.normal_bf16(11, 2, (T, G * Hkv, d))
    first, n = np.asarray(windows, np.int32).T
    B = len(windows)
    table = np.tile(np.arange(pages, dtype=np.int32)[::-1], (B, 1))
    assert Hkv * sum(-(-m * G // 256) for m in n) > Hkv * ((T * G + 255 * B) // 256)
    kv = gcb.KVPool.create(1, Hkv, d, ps, pages)
    kv.planes().copy_(bf16_tensor(pool))
    out = torch.full((T, G * Hkv, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    gcb.gc_prefix_prefill_attn(bf16_tensor(q), kv.handle, _i32(table, "cuda"),
                               _i32(P + first, "cuda"), _i32(n, "cuda"), out, None, 0,
                               _i32(np.append(first, T), "cuda"), B, pages, G * Hkv, d ** -0.5, T)
    assert kv.check() == gcb.GC_OK
    kv.close()
    ref = oracle.prefix_attn(q, pool, 0, table[:1], np.asarray([P], np.int32),
                             np.asarray([0, T], np.int32), d ** -0.5)
    assert_attn_close(out.to(torch.float64).cpu().numpy(), ref, "shared rows")
