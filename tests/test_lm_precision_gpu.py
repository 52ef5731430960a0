"""The LM head of more than 80 sequences on the tensor cores, whose logits were float32 dot products before.

Logits against float64 from the call's own kept states.  A tensor-core accumulator truncates at each of its steps, so what
tells is the bias of the leading logit: with M = 46 from 16 k-blocks of even shares, a segment of one k-block grows to
M / 16 in 4 steps, each losing a quarter of a last place (2^-22 at M / 16) on average: 16 x 4 x 2^-24 = 3.8e-6.  Segments
of two k-blocks lose twice that, so the bound is between the two.
"""
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.bf16 import widen  # noqa: E402
from paper_2609_09338_gb300 import synthetic as syn  # noqa: E402
from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from test_draft_gpu import _built, _dev  # noqa: E402,F401


def draft(B, T):
    """A one-step call of B sequences whose leading logits are 46: its outputs, and its logits in float64."""
    from paper_2609_09338_gb300.binding import to_device_bf16
    from paper_2609_09338_gb300.session import DraftSession
    shape = replace(TINY, d_model=1024, vocab=8192)
    d, V = shape.d_model, shape.vocab
    w = syn.make_weights(shape, 41)
    rng = np.random.default_rng(42)
    embed = widen(w["embed"]) * np.float32(50)
    w["embed"] = syn.bf16_bits(embed)
    w["lm_head"] = syn.bf16_bits(widen(w["lm_head"]) + np.float32(47 / d) * embed[rng.permutation(V)])
    ctx = rng.integers(0, 40, size=B).astype(np.int32)
    kv = syn.make_kv_prefix(shape, ctx, 2, 43)
    di = syn.make_draft_inputs(shape, B, 1, 1, 44)
    sess = DraftSession(shape, w, kv["page_table"], kv["n_pages"], 1)
    sess.append(ctx, kv["k_rows"], kv["v_rows"])
    n0 = sess.kv.seq_len.clone()
    out, kept = sess.draft_buffers(with_logits=True), sess.draft_buffers()
    hidden = torch.zeros((B, 1, d), device="cuda")
    args = (_dev(di["n_new"]), _dev(di["tokens"]), to_device_bf16(di["feats"]), T, _dev(di["u_draft"]))
    sess.draft(*args, out)
    sess.kv.seq_len.copy_(n0)
    sess.draft_hidden(*args, kept, hidden)
    torch.cuda.synchronize()
    assert int(sess.status.item()) == 0
    x = hidden[:, 0].double()
    n = x * torch.rsqrt(x.square().mean(-1, keepdim=True) + shape.rms_eps) * _dev(widen(w["final_norm"])).double()
    z = n @ _dev(widen(w["lm_head"])).double().t()
    assert 44 < float(z.max(-1).values.mean()) < 48
    return out, z


@pytest.mark.parametrize("B", [81, 96, 130])
def test_leading_logits_are_not_biased(B):
    out, z = draft(B, 0.0)
    M, at = z.max(-1)
    got = out["draft_logits"][:, 0].double()
    assert torch.equal(out["draft_tokens"][:, 0].long(), at)
    bias = float((torch.gather(got, 1, at[:, None])[:, 0] - M).mean())
    rms = float((got - z).square().mean().sqrt() / z.square().mean().sqrt())
    assert abs(bias) < 1.4 * 16 * 4 * 2.0 ** -24
    assert rms < 1.6e-7   # the CUDA-core GEMV's


@pytest.mark.parametrize("B", [81, 130])
def test_probabilities_are_those_of_the_logits(B):
    """q(token) = exp(z / T - M) / S with z, M and S of the same sums: a token of nearly all the mass has q = 1 up to the
    rounding of its group's sum, its scaling and the division (a few 2^-24), not 1 + exp(the bias of M)."""
    out, z = draft(B, 0.7)
    tok = out["draft_tokens"][:, 0].long()
    lead = tok == z.argmax(-1)
    assert int(lead.sum()) > B // 2
    q = torch.gather(torch.softmax(z / 0.7, -1), 1, tok[:, None])[:, 0]
    assert float((out["draft_qx"][:, 0].double() / q - 1).abs()[lead].max()) < 8 * 2.0 ** -24
