"""Decode at the batches whose request table brings a block's shared memory to
just below 48 KB, from where on the launch has to ask for more: the static words
of the kernel count too.  The permission outlasts a call, so each variant is the
first of its process to run.  Contexts of 1 to 3 keys of equal value: every
output row is its request's value."""
import subprocess
import sys

import pytest

from paper_2505_23970_gb300 import build as gbuild

pytestmark = pytest.mark.gpu

# (head_dim, q heads per kv head, batch): the last batches for which the dynamic
# part alone stays within 48 KB, per variant of the kernel
WINDOWS = [(128, 8, 5850), (64, 8, 7800), (64, 16, 5560)]

RUN = """
import numpy as np, torch
from paper_2505_23970_gb300 import binding as gcb
d, G, B = {case}
kv = gcb.KVPool.create(1, 1, d, 16, 8)
value = torch.arange(1, 9, device="cuda").view(1, 8, 1, 1, 1)
kv.planes().copy_(value.expand(2, 8, 1, 16, d)[None])
table = (torch.arange(B, dtype=torch.int32, device="cuda") * 5 % 8).view(B, 1)
seq = torch.arange(B, dtype=torch.int32, device="cuda") % 3 + 1
q = torch.ones((B, G, d), dtype=torch.bfloat16, device="cuda")
need = gcb.gc_paged_decode_workspace_bytes(kv.handle, B, 1, G)
ws = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")
image = torch.empty((8, 1, 2, gcb.gc_kv_q8_chunk_bytes(gcb.make_config(1, 1, d, 16, 8))),
                    dtype=torch.uint8, device="cuda")
ids = torch.arange(8, dtype=torch.int32, device="cuda")
gcb.gc_kv_save_q8(kv.handle, image, ids, 8, 0, 1, None, None, gcb.GC_SAVE_DST_DEVICE)
for extra in ([], [image, table, 8, 0]):
    out = torch.zeros_like(q)
    call = gcb.gc_paged_decode_attn_q8 if extra else gcb.gc_paged_decode_attn
    call(q, kv.handle, table, seq, out, None, 0, B, 1, G, d ** -0.5, ws, need, *extra)
    assert kv.check() == gcb.GC_OK
    want = (table + 1).to(torch.bfloat16).view(B, 1, 1).expand_as(out)
    assert torch.equal(out, want)
"""


@pytest.mark.parametrize("case", WINDOWS, ids=str)
def test_first_call_at_the_shared_memory_limit(case):
    gbuild.build()
    r = subprocess.run([sys.executable, "-c", RUN.format(case=case)], cwd=gbuild.ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
