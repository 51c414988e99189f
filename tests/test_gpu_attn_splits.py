"""Prefill attention of calls with few work items at head_dim 128, whose keys
are split over the pairs of a larger cluster (2, 4 or 8 pairs per item):
contexts of fewer steps than pairs (a block table much wider than the
sequence), causal diagonals that cross the parts (rows that see no key of a
part), ragged last steps, a request without prefix and one without new tokens.
Against the float64 oracle, with the suite's tolerance."""
import numpy as np
import pytest

import oracle
from paper_2505_23970_gb300 import binding as gcb
from paper_2505_23970_gb300 import workloads as wl
from paper_2505_23970_gb300.harness import DeviceBatch

from ._util import assert_attn_close

pytestmark = pytest.mark.gpu

CASES = {
    # name: (G, Hkv, ps, prefixes, new tokens, table capacity in tokens)
    "8 pairs": (4, 1, 16, [5000], [43], 0),
    "8 pairs, 8 heads": (8, 8, 16, [7001], [17], 0),
    "4 pairs": (8, 8, 32, [3000, 1411], [30, 1], 0),
    "2 pairs": (8, 4, 16, [900, 77, 1300], [32, 31, 25], 4096),
    "diagonal across parts": (16, 2, 64, [0], [60], 8192),
    "more pairs than steps": (4, 2, 128, [40], [9], 131072),
    "new tokens over several steps": (1, 2, 16, [0, 130], [500, 250], 16384),
    "a request without new tokens": (8, 2, 16, [2000, 600], [0, 9], 4096),
}


@pytest.mark.parametrize("name", list(CASES))
def test_split_matches_oracle(name):
    G, Hkv, ps, P, n, cap = CASES[name]
    w = wl.custom(name, len(P), G * Hkv, Hkv, 128, ps, P, n, seed=len(name))
    wide = max(w.max_blocks, cap // ps)
    w.block_table = np.concatenate(
        [w.block_table, np.full((w.B, wide - w.max_blocks), -1, np.int32)], axis=1)
    db = DeviceBatch(w)
    db.run()
    assert db.check() == gcb.GC_OK
    pool = w.empty_pool()
    if w.prefix_blocks().size:
        oracle.kv_restore(pool, w.host_src(), w.prefix_blocks())
    k, v = w.kv_new()
    oracle.kv_append(pool, 0, k, v, w.block_table, w.prefix_lens, w.cu_new_lens)
    ref = oracle.prefix_attn(w.q(), pool, 0, w.block_table, w.prefix_lens, w.cu_new_lens, w.scale)
    assert_attn_close(db.out_f64(), ref, name)
    first = db.out.clone()
    db.attn()  # the same again: nothing is left over from a launch
    assert db.check() == gcb.GC_OK
    import torch
    assert torch.equal(first.view(torch.int16), db.out.view(torch.int16))
    db.close()


def test_score_jump_in_a_later_part():
    """Keys late in the context score 2^100s above the rest, so the parts'
    reference maxima differ by far more than fp32's range of exponents."""
    w = wl.custom("split-jump", 1, 16, 2, 128, 16, [6000], [20], seed=5)
    q = wl.bf16_bits_to_f32(w.q())
    src = w.host_src()
    for j, h in ((5900, 0), (3001, 1)):
        blk, row = divmod(j, w.ps)
        src[blk, 0, 0, 0, row] = wl.f32_to_bf16_bits(12.0 * q[3, h])
    db = DeviceBatch(w)
    db.run()
    assert db.check() == gcb.GC_OK
    pool = w.empty_pool()
    oracle.kv_restore(pool, src, w.prefix_blocks())
    k, v = w.kv_new()
    oracle.kv_append(pool, 0, k, v, w.block_table, w.prefix_lens, w.cu_new_lens)
    ref = oracle.prefix_attn(w.q(), pool, 0, w.block_table, w.prefix_lens, w.cu_new_lens, w.scale)
    assert_attn_close(db.out_f64(), ref, "split-jump")
    db.close()
