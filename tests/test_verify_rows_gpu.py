"""Streamed verification of rows that are no multiple of 16 bytes (each row at its own misalignment, the last row's end
inside a vector), of the logits-free form, and of tensors whose base is not aligned (the unstreamed kernels), against the
oracle."""
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import verify as ov  # noqa: E402
from paper_2609_09338_gb300 import synthetic as syn  # noqa: E402
from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from parity import check_verify  # noqa: E402
from test_verify_gpu import _built, _oracle, _run  # noqa: E402,F401
from test_verify_hidden_gpu import _inputs, _run_hidden  # noqa: E402


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("V,B,K,T", [(1, 3, 2, 1.0), (5, 9, 3, 0.7), (1025, 7, 3, 1.0), (2049, 6, 4, 0.0), (4097, 5, 2, 1.0),
                                     (4094, 6, 3, 1.0), (40963, 33, 5, 0.7), (2047, 300, 2, 1.0),
                                     (50021, 43, 3, 0.0)])   # (greedy float32 of 32 MB and more: not streamed)
def test_rows_at_any_alignment(V, B, K, T, dtype):
    vi = syn.make_verify_inputs(V, B, K, T, 0.7, seed=V + B + K)
    g, o = _run(vi, T, dtype), _oracle(vi, T, dtype)
    assert check_verify(g["out_tokens"], g["n_accepted"], o, K) <= max(2, B // 8)
    if T > 0:
        np.testing.assert_allclose(g["probs"][..., 0], o["p_x"], atol=1e-5)
        np.testing.assert_allclose(g["probs"][..., 1], o["q_x"], atol=1e-5)


@pytest.mark.parametrize("V,B,K,dtype", [(4099, 9, 3, "f32"), (4097, 6, 3, "bf16"), (8200, 20, 4, "bf16"),
                                         (6145, 83, 2, "bf16"), (2060, 5, 3, "f32")])
def test_without_draft_logits(V, B, K, dtype):
    from paper_2609_09338_gb300 import binding as ob
    shape = replace(TINY, vocab=V)
    w = syn.make_weights(shape, seed=V + B)
    ctx = ob.osprey_create(shape, ob.upload_weights(w))
    inp = _inputs(shape, w, B, K, 1.0, 0.7, seed=V + K)
    g = _run_hidden(ctx, inp, 1.0, dtype)
    assert g["status"] == 0
    o = ov.verify_hidden(inp["target"] if dtype == "f32" else syn.bf16_bits(inp["target"]), inp["hidden"], w["lm_head"],
                         w["final_norm"], shape.rms_eps, inp["x"], 1.0, inp["u_accept"], inp["u_sample"])
    check_verify(g["out_tokens"], g["n_accepted"], o, K)
    np.testing.assert_allclose(g["probs"][..., 0], o["p_x"], atol=1e-5)
    np.testing.assert_array_equal(g["probs"][..., 1], inp["qx"])


def test_unaligned_base():
    """A view one element into its buffer takes the unstreamed kernels and gives the same tokens."""
    from paper_2609_09338_gb300.session import VerifyBuffers
    V, B, K = 3001, 4, 3
    vi = syn.make_verify_inputs(V, B, K, 1.0, 0.7, seed=5)
    want = _run(vi, 1.0)

    def shifted(a):
        buf = torch.empty(a.size + 1, device="cuda")
        buf[1:] = torch.from_numpy(a).cuda().reshape(-1)
        return buf[1:].view(a.shape)

    vb = VerifyBuffers(B, K, V)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    vb.run(shifted(vi["target_logits"]), shifted(vi["draft_logits"]), dev(vi["draft_tokens"]), 1.0, dev(vi["u_accept"]),
           dev(vi["u_sample"]))
    torch.cuda.synchronize()
    assert int(vb.status.item()) == 0
    np.testing.assert_array_equal(vb.n_accepted.cpu().numpy(), want["n_accepted"])
    np.testing.assert_array_equal(vb.out_tokens.cpu().numpy(), want["out_tokens"])
