"""Decode attention at the edges of its work splits: contexts around a group
of 16 keys, around the longest context of the pair-per-warp split, shares that
cut a pair at odd places, pieces with more groups per warp than one block of
look-ups holds.  Long contexts repeat the pages of a small pool (the kernel
only reads through the block table), so the float64 oracle stays cheap; the
tolerance is the suite's (bf16 P and output).  With `q8`, every other page of a
context comes from the 8-bit image and the result is also bit for bit that of
the same call on the restored pool."""
import numpy as np
import pytest

import oracle
from paper_2505_23970_gb300 import binding as gcb
from paper_2505_23970_gb300 import workloads as wl
from paper_2505_23970_gb300.harness import _i32, bf16_tensor

from ._util import assert_attn_close

pytestmark = pytest.mark.gpu

PAGES = 64


def _around(*edges):
    return [t for e in edges for t in (e - 1, e, e + 1) if t > 0]


CASES = {
    # name: (G, Hkv, d, ps, context lengths)
    "groups": (4, 2, 128, 16, _around(1, 16, 32, 96, 192)),
    "pair-per-warp": (8, 8, 128, 16, [256, 1, 255, 17] + [t % 250 + 3 for t in range(116)]),
    "one-above-short": (8, 8, 128, 16, [257, 1, 255, 17] + [t % 250 + 3 for t in range(116)]),
    "pair-per-warp-d64-g16": (16, 16, 64, 32, [256, 1, 15, 33] + [t % 250 + 3 for t in range(92)]),
    "ranges-d64": (2, 2, 64, 16, _around(512, 2048) + [5000]),
    "shares-g16": (16, 2, 128, 64, _around(192, 4096) + [9999]),
    "cut-odd": (8, 1, 128, 16, [7001, 333, 58000]),
    "many-look-ups": (1, 8, 128, 128, [125001]),
    # share boundaries at every place of a pair and of the allowance in front of it
    "cut-anywhere": (8, 8, 128, 16, [16 * (1 + t % 40) for t in range(96)]),
    "short-and-long": (4, 2, 128, 32, [1] * 60 + [20000] + [2, 300] * 20),
}


@pytest.mark.parametrize("q8", [False, True])
@pytest.mark.parametrize("name", list(CASES))
def test_decode_split(name, q8):
    import torch
    G, Hkv, d, ps, ctx = CASES[name]
    rng = np.random.default_rng(len(name))
    B, Hq = len(ctx), G * Hkv
    seq = np.asarray(ctx, np.int32)
    width = -(-max(ctx) // ps)
    table = rng.integers(0, PAGES, size=(B, width)).astype(np.int32)
    pool = wl.normal_bf16(7, 1, (1, 2, PAGES, Hkv, ps, d))
    q = wl.normal_bf16(7, 2, (B, Hq, d))
    scale = d ** -0.5
    kv = gcb.KVPool.create(1, Hkv, d, ps, PAGES)
    image = mapped = None
    if q8:
        # image block i holds page i; odd pages of a context are read from it
        ids = np.arange(PAGES, dtype=np.int32)
        image = oracle.kv_save_q8(pool, ids)
        restored = pool.copy()
        oracle.kv_restore_q8(restored, image, ids)
        mapped = np.where(np.arange(width)[None] % 2 == 1, table, -1).astype(np.int32)
        # the pages read from the pool hold the same values
        pool = restored
    kv.planes().copy_(bf16_tensor(pool))
    dq, dt, ds = bf16_tensor(q), _i32(table, "cuda"), _i32(seq, "cuda")
    need = gcb.gc_paged_decode_workspace_bytes(kv.handle, B, width, Hq)
    ws = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")
    out = torch.full((B, Hq, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    gcb.gc_paged_decode_attn(dq, kv.handle, dt, ds, out, None, 0, B, width, Hq, scale, ws, need)
    assert kv.check() == gcb.GC_OK
    if q8:
        same = torch.full_like(out, float("nan"))
        gcb.gc_paged_decode_attn_q8(dq, kv.handle, dt, ds, same, None, 0, B, width, Hq, scale, ws,
                                    need, torch.from_numpy(image).cuda(), _i32(mapped, "cuda"),
                                    PAGES, 0)
        assert kv.check() == gcb.GC_OK
        assert torch.equal(out.view(torch.int16), same.view(torch.int16)), name
    ref = oracle.prefix_attn(q, pool, 0, table, seq - 1, np.arange(B + 1, dtype=np.int32), scale)
    assert_attn_close(out.to(torch.float64).cpu().numpy(), ref, name)
    kv.close()


@pytest.mark.parametrize("B,width,longest", [(256, 131072, 3000), (8192, 32767, 300)],
                         ids=["units of 128 keys", "no allowance"])
def test_wide_tables(B, width, longest):
    """Tables so wide that the units of 16 keys, then also the allowance in front
    of a pair, could not be counted in 32 bits if every context filled its own."""
    import torch
    Hkv, d, ps, pages = 8, 128, 128, 16
    assert B * Hkv * (width * ps // 16) >= 2**31 - 448
    rng = np.random.default_rng(B)
    seq = rng.integers(1, longest, size=B, endpoint=True).astype(np.int32)
    near = -(-longest // ps)
    table = rng.integers(0, pages, size=(B, near)).astype(np.int32)
    pool = wl.normal_bf16(5, 1, (1, 2, pages, Hkv, ps, d))
    q = wl.normal_bf16(5, 2, (B, Hkv, d))
    kv = gcb.KVPool.create(1, Hkv, d, ps, pages)
    kv.planes().copy_(bf16_tensor(pool))
    wide = torch.full((B, width), -1, dtype=torch.int32, device="cuda")
    wide[:, :near] = _i32(table, "cuda")
    need = gcb.gc_paged_decode_workspace_bytes(kv.handle, B, width, Hkv)
    ws = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")
    out = torch.full((B, Hkv, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    gcb.gc_paged_decode_attn(bf16_tensor(q), kv.handle, wide, _i32(seq, "cuda"), out, None, 0, B,
                             width, Hkv, d ** -0.5, ws, need)
    assert kv.check() == gcb.GC_OK
    kv.close()
    ref = oracle.prefix_attn(q, pool, 0, table, seq - 1, np.arange(B + 1, dtype=np.int32),
                             d ** -0.5)
    assert_attn_close(out.to(torch.float64).cpu().numpy(), ref, "wide table")


@pytest.mark.parametrize("d,Hkv,pages", [(128, 1, 3000), (128, 2, 1200), (64, 1, 700)])
def test_leading_pages_invalid(d, Hkv, pages):
    """Bad block-table entries are left out and recorded; also where they fill the
    first pieces of a context cut over many (more than the merge takes at a time)."""
    import torch
    ps, bad, G = 16, pages * 2 // 3, 8
    rng = np.random.default_rng(pages)
    table = rng.integers(0, PAGES, size=(2, pages)).astype(np.int32)
    seq = np.asarray([pages * ps - 5, pages * ps - 77], np.int32)
    pool = wl.normal_bf16(9, 1, (1, 2, PAGES, Hkv, ps, d))
    q = wl.normal_bf16(9, 2, (2, G * Hkv, d))
    kv = gcb.KVPool.create(1, Hkv, d, ps, PAGES)
    kv.planes().copy_(bf16_tensor(pool))
    given = table.copy()
    given[:, :bad] = -1
    need = gcb.gc_paged_decode_workspace_bytes(kv.handle, 2, pages, G * Hkv)
    ws = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")
    out = torch.full((2, G * Hkv, d), float("nan"), dtype=torch.bfloat16, device="cuda")
    gcb.gc_paged_decode_attn(bf16_tensor(q), kv.handle, _i32(given, "cuda"), _i32(seq, "cuda"),
                             out, None, 0, 2, pages, G * Hkv, d ** -0.5, ws, need)
    assert kv.check() == gcb.GC_ERR_OUT_OF_RANGE
    assert kv.check() == gcb.GC_OK
    kv.close()
    ref = oracle.prefix_attn(q, pool, 0, np.ascontiguousarray(table[:, bad:]),
                             seq - bad * ps - 1, np.arange(3, dtype=np.int32), d ** -0.5)
    assert_attn_close(out.to(torch.float64).cpu().numpy(), ref, "leading pages invalid")
