"""The two routes of gc_prefix_prefill_attn_q8: image pages dequantised once
into scratch and then read like pool pages, and (while the stream is being
captured, when there is no scratch) dequantised by the attention kernel.  Both
against the float64 oracle with the suite's tolerance, bit for bit the same as
each other at head_dim 64, where the tiles and their order are the same.
Scratch pages are numbered by image block, or by table position when the image
has more blocks than the table has entries."""
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2505_23970_gb300 import binding as gcb
from paper_2505_23970_gb300 import build as gbuild
from paper_2505_23970_gb300 import workloads as wl
from paper_2505_23970_gb300.harness import DeviceBatch, _i32

from ._q8 import Q8Case
from ._util import assert_attn_close

pytestmark = pytest.mark.gpu

CASES = {
    # name: (G, Hkv, d, ps, prefixes, new tokens, unused image blocks in front)
    "d128": (8, 2, 128, 16, [300, 0, 1000, 17], [70, 45, 0, 260], 0),
    "d128 by position": (4, 1, 128, 32, [700, 129], [33, 1], 5000),
    "d128 one head, split": (8, 1, 128, 128, [5000], [9], 1),
    "d64": (4, 3, 64, 16, [301, 0, 990, 64], [70, 129, 0, 260], 0),
    "d64 by position": (16, 1, 64, 64, [640, 65], [5, 200], 300),
}


def _call(db, w, image, table, n, stream):
    gcb.gc_prefix_prefill_attn_q8(db.q, db.pool.handle, db.block_table, db.prefix_lens,
                                  db.new_lens, db.out, stream, 0, db.cu_new_lens, w.B,
                                  w.max_blocks, w.Hq, w.scale, w.T_new, image, table, n, 0)


def _batch(w, case):
    """The batch's pool with what the 8-bit table leaves to it: partly cached pages
    and the new tokens."""
    import torch
    db = DeviceBatch(w, with_restore=False)
    if case.to_pool.size:
        part = torch.from_numpy(np.ascontiguousarray(case.img[case.to_pool])).cuda()
        gcb.gc_kv_restore_q8(db.pool.handle, part, _i32(case.ids[case.to_pool], "cuda"),
                             int(case.to_pool.size), 0, w.L, None, None,
                             gcb.GC_RESTORE_SRC_DEVICE)
    db.append(layer=0)
    return db


def _both_routes(db, w, image, table, n):
    import torch
    _call(db, w, image, table, n, None)
    assert db.check() == gcb.GC_OK
    eager = db.out.clone()
    db.out.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _call(db, w, image, table, n, torch.cuda.current_stream().cuda_stream)
    graph.replay()
    torch.cuda.synchronize()
    assert db.check() == gcb.GC_OK
    return eager, db.out.clone()


@pytest.mark.parametrize("name", list(CASES))
def test_routes_match_oracle(name):
    import torch
    G, Hkv, d, ps, P, n, spare = CASES[name]
    w = wl.custom(name, len(P), G * Hkv, Hkv, d, ps, P, n, seed=len(name))
    case = Q8Case(w, frac_in_image=0.8, seed=1)
    db = _batch(w, case)
    img = torch.from_numpy(case.img).cuda()
    img = torch.cat([torch.full((spare, *img.shape[1:]), 0xFF, dtype=img.dtype, device="cuda"), img])
    table = _i32(np.where(case.table >= 0, case.table + spare, -1), "cuda")
    out = _both_routes(db, w, img, table, int(img.shape[0]))
    db.close()
    if d == 64:
        assert torch.equal(out[0].view(torch.int16), out[1].view(torch.int16))
    ref = oracle.prefix_attn(w.q(), case.oracle_pool(), 0, w.block_table, w.prefix_lens,
                             w.cu_new_lens, w.scale)
    for o, route in zip(out, ("scratch", "captured")):
        assert_attn_close(o.to(torch.float64).cpu().numpy(), ref, f"{name} [{route}]")


def test_image_blocks_shared_by_requests():
    """Two requests naming the same image blocks give what two copies of the
    blocks give."""
    import torch
    w = wl.custom("shared", 2, 16, 2, 128, 16, [640, 640], [40, 40], seed=4)
    case = Q8Case(w)
    full = 640 // 16
    case.img[full:2 * full] = case.img[:full]
    db = DeviceBatch(w, with_restore=False)
    db.append(layer=0)
    img = torch.from_numpy(case.img).cuda()
    shared = case.table.copy()
    shared[1, :full] = shared[0, :full]
    outs = []
    for t in (case.table, shared):
        _call(db, w, img, _i32(t, "cuda"), int(img.shape[0]), None)
        assert db.check() == gcb.GC_OK
        outs.append(db.out.clone())
    db.close()
    assert torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))


RESET = """
import ctypes, os, re
import torch
from paper_2505_23970_gb300 import binding as gcb
torch.cuda.init()
cudart = next(l.split()[-1] for l in open("/proc/self/maps") if re.search(r"libcudart\\.so", l))
rt = ctypes.CDLL(cudart)
cfg = gcb.make_config(1, 1, 128, 16, 4)
size = gcb.gc_kv_pool_bytes(cfg)

def pool():
    p = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
    return gcb.gc_kv_pool_create(cfg, p.value, size)

first, second = pool(), pool()
assert rt.cudaDeviceReset() == 0
gcb.gc_kv_pool_destroy(first)      # no newer pool
third = pool()
gcb.gc_kv_pool_destroy(second)     # next to a newer one
fourth = pool()
gcb.gc_kv_pool_destroy(third)
gcb.gc_kv_pool_destroy(fourth)
assert rt.cudaDeviceSynchronize() == 0
print("done", flush=True)
os._exit(0)
"""


def test_pools_destroyed_after_a_device_reset():
    """A pool in caller-owned memory outlives its context: destroying it later
    touches neither the allocator that the reset took nor the next context's."""
    r = subprocess.run([sys.executable, "-c", RESET], cwd=gbuild.ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["done"], r.stderr[-2000:]


def _tight_call(w, seed):
    """A batch, its image and table on the GPU, and the result on the default stream."""
    import torch
    case = Q8Case(w, seed=seed)
    db = _batch(w, case)
    img, table = torch.from_numpy(case.img).cuda(), _i32(case.table, "cuda")
    _call(db, w, img, table, int(img.shape[0]), None)
    assert db.check() == gcb.GC_OK and torch.isfinite(db.out).all()
    return db, img, table, db.out.clone()


def test_more_pages_than_scratch_may_hold():
    """An image of more blocks, and tables of more entries, than 1 GiB of scratch
    has pages: the second route is taken, as under capture, with its result."""
    import torch
    w = wl.custom("no scratch", 4, 16, 8, 128, 16, [640, 33, 1000, 512], [40, 300, 1, 77], seed=6)
    case = Q8Case(w)
    db = _batch(w, case)
    wide, blocks = 4200, 16400  # pages of 32 KB per plane
    assert min(4 * wide, blocks) * 2 * 8 * 16 * 128 * 2 > 1 << 30
    image = torch.zeros((blocks, *case.img.shape[1:]), dtype=torch.uint8, device="cuda")
    image[-case.img.shape[0]:] = torch.from_numpy(case.img).cuda()
    shift = blocks - case.img.shape[0]

    def widen(t):
        t = np.concatenate([t, np.full((4, wide - t.shape[1]), -1, t.dtype)], axis=1)
        return _i32(t, "cuda")
    bt, qt = widen(w.block_table), widen(np.where(case.table >= 0, case.table + shift, -1))

    def call(stream):
        gcb.gc_prefix_prefill_attn_q8(db.q, db.pool.handle, bt, db.prefix_lens, db.new_lens,
                                      db.out, stream, 0, db.cu_new_lens, w.B, wide, w.Hq, w.scale,
                                      w.T_new, image, qt, blocks, 0)
    call(None)
    assert db.check() == gcb.GC_OK
    eager = db.out.clone()
    db.out.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(torch.cuda.current_stream().cuda_stream)
    graph.replay()
    torch.cuda.synchronize()
    assert db.check() == gcb.GC_OK
    assert torch.equal(eager.view(torch.int16), db.out.view(torch.int16))
    db.close()
    ref = oracle.prefix_attn(w.q(), case.oracle_pool(), 0, w.block_table, w.prefix_lens,
                             w.cu_new_lens, w.scale)
    assert_attn_close(eager.to(torch.float64).cpu().numpy(), ref, "no scratch")


def test_pools_on_their_own_streams_and_threads():
    """Two pools of a device share the scratch allocator, not the scratch: calls of
    two threads on two streams give what each gives alone."""
    import threading

    import torch
    works = [wl.custom("left", 3, 16, 2, 128, 16, [2000, 700, 64], [70, 200, 30], seed=7),
             wl.custom("right", 2, 8, 2, 128, 16, [3000, 31], [150, 40], seed=8)]
    calls = [_tight_call(w, 9) for w in works]
    torch.cuda.synchronize()
    wrong = []

    def loop(w, db, img, table, want):
        stream = torch.cuda.Stream()
        for _ in range(60):
            with torch.cuda.stream(stream):
                db.out.zero_()
                _call(db, w, img, table, int(img.shape[0]), stream.cuda_stream)
                if not torch.equal(db.out.view(torch.int16), want.view(torch.int16)):
                    wrong.append(w.name)
    threads = [threading.Thread(target=loop, args=(w, *c)) for w, c in zip(works, calls)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    for db, *_ in calls:
        assert db.check() == gcb.GC_OK
        db.close()
