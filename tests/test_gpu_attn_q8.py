"""Prefill over pages kept in the 8-bit cache tier (gc_prefix_prefill_attn_q8).

The operation is defined as the 8-bit restore (Sec. 6.1 keeps the 70B KV in
INT8) followed by prefix-reuse attention (Sec. 2.2), so the oracle is
oracle.kv_restore_q8 of every cached page, oracle.kv_append and
oracle.prefix_attn.  The GPU path never writes the 8-bit pages into the
pool.  Each call is made on both routes: as the library chooses, which for most
of these sizes dequantises the pages once into scratch, and captured into a
graph, where the single-SM kernel's 8-bit variant dequantises them itself.  Both
are checked against the library's own two-step path (gc_kv_restore_q8 of every
page, then gc_prefix_prefill_attn): bit for bit at head_dim 64, where all of them
run on the same single-SM kernel, and within the attention tolerance at head_dim
128, where the two-step path runs on SM pairs; and within the attention tolerance
against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2505_23970_gb300 import binding as gcb
from paper_2505_23970_gb300 import workloads as wl
from paper_2505_23970_gb300.harness import DeviceBatch, _i32

from ._q8 import Q8Case, all_pages_case
from ._util import assert_attn_close, gather_rows, sample_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2505_23970_gb300 import build
    build.build()


def _dev_image(img, layer_major):
    import torch
    if layer_major:
        img = np.ascontiguousarray(img.swapaxes(0, 1))
    return torch.from_numpy(img).cuda()


def on_route(call, captured):
    """Make the call now, or captured into a graph that is then run."""
    import torch
    if not captured:
        call(None)
        return
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(torch.cuda.current_stream().cuda_stream)
    graph.replay()
    torch.cuda.synchronize()


def run_q8(case, layer=0, layer_major=False, table=None, captured=False):
    """Restore the pool-side pages, append, attention over the q8 table."""
    import torch
    w = case.w
    db = DeviceBatch(w, with_restore=False)
    if case.to_pool.size:
        part = torch.from_numpy(np.ascontiguousarray(case.img[case.to_pool])).cuda()
        gcb.gc_kv_restore_q8(db.pool.handle, part, _i32(case.ids[case.to_pool], "cuda"),
                             int(case.to_pool.size), 0, w.L, None, None,
                             gcb.GC_RESTORE_SRC_DEVICE)
    for l in range(w.L):
        db.append(layer=l)
    dimg = _dev_image(case.img, layer_major)
    flags = gcb.GC_RESTORE_LAYER_MAJOR if layer_major else 0
    dtab = _i32(case.table if table is None else table, "cuda")
    on_route(lambda stream: gcb.gc_prefix_prefill_attn_q8(
        db.q, db.pool.handle, db.block_table, db.prefix_lens, db.new_lens, db.out, stream, layer,
        db.cu_new_lens, w.B, w.max_blocks, w.Hq, w.scale, w.T_new, dimg, dtab, int(case.ids.size),
        flags), captured)
    status = db.check()
    out = db.out.clone()
    pool = db.pool_bits()
    db.close()
    return status, out, pool


def run_restore_then_attn(case, layer=0):
    """The two-step path: every cached page dequantised into the pool."""
    import torch
    w = case.w
    db = DeviceBatch(w, with_restore=False)
    if case.ids.size:
        gcb.gc_kv_restore_q8(db.pool.handle, torch.from_numpy(case.img).cuda(),
                             _i32(case.ids, "cuda"), int(case.ids.size), 0, w.L, None, None,
                             gcb.GC_RESTORE_SRC_DEVICE)
    for l in range(w.L):
        db.append(layer=l)
    db.attn(layer=layer)
    assert db.check() == gcb.GC_OK
    out = db.out.clone()
    db.close()
    return out


def _bits_equal(a, b):
    import torch
    return torch.equal(a.view(torch.int16), b.view(torch.int16))


def same_as_two_step(w, out, two_step, what, rows=None):
    """Bit for bit at head_dim 64 (both on the single-SM kernel); within the
    attention tolerance at 128 (the two-step path runs on SM pairs)."""
    import torch
    if w.d == 64:
        assert _bits_equal(out, two_step), f"{what}: differs from restore + attn"
        return
    a = out.to(torch.float64).cpu().numpy()
    b = two_step.to(torch.float64).cpu().numpy()
    if rows is not None:
        a, b = gather_rows(a, w, rows), gather_rows(b, w, rows)
    assert_attn_close(a, b, f"{what} vs restore + attn")


def full_q8_parity(w, **kw):
    import torch
    case = Q8Case(w, **kw)
    two_step = run_restore_then_attn(case)
    ref = oracle.prefix_attn(w.q(), case.oracle_pool(), 0, w.block_table, w.prefix_lens,
                             w.cu_new_lens, w.scale)
    for captured in (False, True):
        status, out, _ = run_q8(case, captured=captured)
        assert status == gcb.GC_OK
        same_as_two_step(w, out, two_step, w.name)
        assert_attn_close(out.to(torch.float64).cpu().numpy(), ref, f"{w.name} [q8, {captured}]")


def sampled_q8_parity(w, n_random=512):
    import torch
    case = Q8Case(w)
    rows = sample_rows(w, n_random)
    two_step = run_restore_then_attn(case)
    ref = oracle.prefix_attn_rows(w.q(), case.oracle_pool(), 0, w.block_table, w.prefix_lens,
                                  w.cu_new_lens, w.scale, rows)
    for captured in (False, True):
        status, out, _ = run_q8(case, captured=captured)
        assert status == gcb.GC_OK
        same_as_two_step(w, out, two_step, w.name, rows)
        got = gather_rows(out.to(torch.float64).cpu().numpy(), w, rows)
        assert_attn_close(got, ref, f"{w.name} sampled [q8, {captured}]")


# ---------------------------------------------------------------- shapes
@pytest.mark.parametrize("G,d,ps", [(8, 128, 16), (4, 64, 16), (1, 128, 32), (16, 64, 64),
                                    (2, 128, 128)])
def test_q8_shapes_ragged(G, d, ps):
    """Head groupings, both head sizes and every page size, with prefixes
    that end inside a page, a request without prefix and one without new
    tokens: against restore + attention (bit for bit at head_dim 64) and
    within tolerance of the oracle."""
    Hkv = 2
    w = wl.custom(f"q8-G{G}-d{d}-ps{ps}", 5, G * Hkv, Hkv, d, ps, [300, 0, 1000, 17, 640],
                  [70, 45, 0, 260, 129], seed=G * 7 + d + ps)
    full_q8_parity(w)


def test_q8_tiny():
    full_q8_parity(wl.tiny())


def test_q8_mixed_pool_and_image_pages():
    """Half of the full prefix pages read from the image, the other half
    already in the pool: the kernel takes each page from where the table
    says, with the same result as the all-pool path."""
    w = wl.custom("q8-mixed", 3, 16, 2, 128, 16, [2000, 700, 129], [200, 64, 300], seed=31)
    full_q8_parity(w, frac_in_image=0.5, seed=3)


def test_q8_llama3_70b_layer_sampled():
    """The 70B-shaped layer (8 x (8192 cached + 1024 new), 64/8 heads)."""
    sampled_q8_parity(wl.llama3_70b_layer())


def test_q8_conversation_mix_sampled():
    """The multi-turn mix (64 requests, lognormal lengths, every prefix hit)."""
    sampled_q8_parity(wl.conversation_mix(hit_p=1.0))


def test_q8_long_document_sampled():
    """131072 cached tokens in 64-token pages."""
    sampled_q8_parity(wl.long_document(B=1), n_random=128)


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("layer_major", [False, True])
def test_q8_layer_of_a_multilayer_image(layer_major, captured):
    """An image of three layers, attention of layer 1, in both image
    layouts: only layer 1's chunks are read."""
    w = wl.custom("q8-layers", 2, 16, 2, 128, 16, [520, 47], [40, 129], seed=15)
    w.L = 3
    case = Q8Case(w)
    status, out, _ = run_q8(case, layer=1, layer_major=layer_major, captured=captured)
    assert status == gcb.GC_OK
    same_as_two_step(w, out, run_restore_then_attn(case, layer=1), "layer 1")
    import torch
    ref = oracle.prefix_attn(w.q(), case.oracle_pool(), 1, w.block_table, w.prefix_lens,
                             w.cu_new_lens, w.scale)
    assert_attn_close(out.to(torch.float64).cpu().numpy(), ref, "layer 1 [q8]")


@pytest.mark.parametrize("captured", [False, True])
def test_q8_pool_pages_of_image_pages_are_not_read(captured):
    """Pool pages behind image-mapped table entries keep their NaN fill
    (nothing restores them) and the pool is not written by the call."""
    w = wl.custom("q8-untouched", 2, 16, 2, 128, 16, [640, 300], [64, 20], seed=9)
    case = Q8Case(w)
    status, out, pool = run_q8(case, captured=captured)
    assert status == gcb.GC_OK
    import torch
    assert torch.isfinite(out.float()).all()
    for b in range(w.B):
        for j in range(w.max_blocks):
            if case.table[b, j] >= 0:
                page = w.block_table[b, j]
                assert np.all(pool[0, :, page] == 0x7FC0)


@pytest.mark.parametrize("captured", [False, True])
def test_q8_bad_table_entry_is_reported_not_faulted(captured):
    """An image block >= n_image_blocks is skipped and recorded as
    GC_ERR_OUT_OF_RANGE in the status word."""
    w = wl.custom("q8-bad", 2, 16, 2, 128, 16, [640, 300], [64, 20], seed=10)
    case = Q8Case(w)
    bad = case.table.copy()
    bad[1, 2] = case.ids.size + 5
    status, _, _ = run_q8(case, table=bad, captured=captured)
    assert status == gcb.GC_ERR_OUT_OF_RANGE


def test_q8_host_checks():
    """Unknown flags, a NULL table and a misaligned image fail before any
    launch with GC_ERR_INVALID_ARG."""
    import torch
    w = wl.custom("q8-args", 1, 16, 2, 128, 16, [64], [16], seed=11)
    case = Q8Case(w)
    db = DeviceBatch(w, with_restore=False)
    dimg = _dev_image(case.img, False)
    tab = _i32(case.table, "cuda")
    args = (db.q, db.pool.handle, db.block_table, db.prefix_lens, db.new_lens, db.out, None, 0,
            db.cu_new_lens, w.B, w.max_blocks, w.Hq, w.scale, w.T_new)
    for image, table, flags in ((dimg, tab, 0x10), (dimg, None, 0),
                                (dimg.data_ptr() + 4, tab, 0)):
        with pytest.raises(gcb.GcError) as e:
            gcb.gc_prefix_prefill_attn_q8(*args, image, table, int(case.ids.size), flags)
        assert e.value.status == gcb.GC_ERR_INVALID_ARG
    torch.cuda.synchronize()
    db.close()


@pytest.mark.parametrize("captured", [False, True])
@pytest.mark.parametrize("d", [128, 64])
def test_q8_every_page_from_the_image(d, captured):
    """Sequences that end inside an image page: V rows past the end are
    zeroed, under capture by the converters (the pool holds NaN everywhere),
    keys past the end are masked; against restore + attention (bit for bit at
    head_dim 64) and the oracle."""
    import torch
    w = wl.custom(f"q8-allimg-d{d}", 4, 16, 2, d, 16, [300, 0, 77, 640], [70, 45, 3, 129],
                  seed=17 + d)
    img, ids, table, ref_pool = all_pages_case(w)
    db = DeviceBatch(w, with_restore=False)
    dimg = torch.from_numpy(img).cuda()
    dtab = _i32(table, "cuda")
    on_route(lambda stream: gcb.gc_prefix_prefill_attn_q8(
        db.q, db.pool.handle, db.block_table, db.prefix_lens, db.new_lens, db.out, stream, 0,
        db.cu_new_lens, w.B, w.max_blocks, w.Hq, w.scale, w.T_new, dimg, dtab, int(ids.size), 0),
        captured)
    assert db.check() == gcb.GC_OK
    out = db.out.clone()
    db.close()
    db = DeviceBatch(w, with_restore=False)
    gcb.gc_kv_restore_q8(db.pool.handle, dimg, _i32(ids, "cuda"), int(ids.size), 0, w.L, None,
                         None, gcb.GC_RESTORE_SRC_DEVICE)
    db.attn()
    assert db.check() == gcb.GC_OK
    same_as_two_step(w, out, db.out, w.name)
    db.close()
    ref = oracle.prefix_attn(w.q(), ref_pool, 0, w.block_table, w.prefix_lens, w.cu_new_lens,
                             w.scale)
    assert_attn_close(out.to(torch.float64).cpu().numpy(), ref, f"{w.name} [q8, all pages]")


def test_q8_largest_batch():
    """8192 requests through the 16-warp variant (its 8-bit state sits after
    the unit table in shared memory)."""
    rng = np.random.default_rng(43)
    B = 8192
    w = wl.custom("q8-batch-8192", B, 4, 2, 128, 16, rng.integers(0, 80, size=B),
                  rng.integers(0, 4, size=B), seed=43)
    full_q8_parity(w)
