"""A process's first draft call on the tensor cores, captured into a CUDA graph without a call before it: the kernels are
opted into their shared memory at their first launch, which a capture has to allow."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CODE = """
import sys
import numpy as np, torch
from paper_2609_09338_gb300 import synthetic as syn
from paper_2609_09338_gb300.binding import to_device_bf16
from paper_2609_09338_gb300.session import DraftSession
from paper_2609_09338_gb300.workloads import TINY
B = int(sys.argv[1])
ctx = np.arange(B, dtype=np.int32) % 40
kv = syn.make_kv_prefix(TINY, ctx, 4, 1)
di = syn.make_draft_inputs(TINY, B, 1, 3, 2)
sess = DraftSession(TINY, syn.make_weights(TINY, 3), kv["page_table"], kv["n_pages"], 3, 1)
sess.append(ctx, kv["k_rows"], kv["v_rows"])
dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
args = (dev(di["n_new"]), dev(di["tokens"]), to_device_bf16(di["feats"]), 1.0, dev(di["u_draft"]))
out = [sess.draft_buffers(with_logits=True) for _ in range(2)]
n0 = sess.kv.seq_len.clone()
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    sess.draft(*args, out[0])
g.replay()
torch.cuda.synchronize()
sess.kv.seq_len.copy_(n0)   # a call commits its new rows
sess.draft(*args, out[1])
torch.cuda.synchronize()
assert int(sess.status.item()) == 0
assert all(torch.equal(out[0][k], out[1][k]) for k in out[0] if out[0][k] is not None)
print("captured")
"""


@pytest.mark.parametrize("B", [3, 96])
def test_first_call_captured(B):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE, str(B)], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stderr[-2000:]
