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
    db = DeviceBatch(w, with_restore=False)
    if case.to_pool.size:
        part = torch.from_numpy(np.ascontiguousarray(case.img[case.to_pool])).cuda()
        gcb.gc_kv_restore_q8(db.pool.handle, part, _i32(case.ids[case.to_pool], "cuda"),
                             int(case.to_pool.size), 0, w.L, None, None,
                             gcb.GC_RESTORE_SRC_DEVICE)
    db.append(layer=0)
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
