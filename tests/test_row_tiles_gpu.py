"""Draft calls of more than 80 rows: the tensor-core projections and the LM head run in tiles of rows.

Sizes at the edges of the tiling (one row past a tile, a last tile that is nearly empty, several tiles, ragged extend
rows), against the oracle with the tolerances of the other draft tests.
"""
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2609_09338_gb300 import synthetic as syn  # noqa: E402
from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from test_draft_gpu import _built, check_case, run_case  # noqa: E402,F401


@pytest.mark.parametrize("B,max_new,T", [(81, 1, 0.0), (96, 1, 1.0), (161, 1, 0.0), (27, 3, 0.0), (33, 8, 1.0)])
def test_more_rows_than_a_tile(B, max_new, T):
    rng = np.random.default_rng(B)
    ctx = rng.integers(0, 40, size=B)
    n_new = rng.integers(1, max_new + 1, size=B)
    pick = sorted({0, B // 2, B - 1, min(79, B - 1), min(80, B - 1)})
    check_case(run_case(TINY, ctx, 3, T, 50 + B, n_new=n_new, max_new=max_new, peaked=T > 0, sample_seqs=pick))


@pytest.mark.parametrize("B,max_new", [(81, 1), (129, 1), (27, 8)])
def test_long_reductions(B, max_new):
    """Reductions of 4096 take the larger tiles (one CTA per SM), their neighbours of a layer the small ones: the operand
    planes between them have either's rows."""
    shape = replace(TINY, ffn_dim=4096, feat_dim=4096, n_layers=2)
    rng = np.random.default_rng(B)
    n_new = rng.integers(1, max_new + 1, size=B)
    pick = sorted({0, B // 2, B - 1, min(80, B - 1)})
    check_case(run_case(shape, rng.integers(0, 30, size=B), 2, 0.0, 30 + B, n_new=n_new, max_new=max_new, sample_seqs=pick))


@pytest.mark.parametrize("d", [1792, 2048, 2304, 3840, 4096])
def test_wide_rows(d):
    """The blocks that normalise and gather rows are wider from d 2048 and from d 4096: both sides of each edge, a last
    pass that is partly filled, ragged extend rows."""
    shape = replace(TINY, d_model=d)
    n_new = np.array([1, 3, 2, 3])
    check_case(run_case(shape, np.array([5, 0, 17, 30]), 2, 0.0, 90 + d, n_new=n_new, max_new=3))


def test_block_rows_beyond_a_tile():
    """Ten blocks of 11 positions (100 rows: two row tiles, groups of 8 and 2 sequences) give what each gives in a call of
    its own."""
    from paper_2609_09338_gb300.binding import to_device_bf16
    from paper_2609_09338_gb300.session import DflashSession
    B, block = 10, 11
    P = block - 1
    rng = np.random.default_rng(3)
    ctx = rng.integers(1, 50, size=B).astype(np.int32)
    w = syn.make_weights(TINY, 71)
    kv = syn.make_kv_prefix(TINY, ctx, P, 72)
    anchors = rng.integers(0, TINY.vocab, size=B).astype(np.int32)
    feats = syn.make_draft_inputs(TINY, B, 1, 1, 73)["feats"][:, 0]
    offs = np.concatenate([[0], np.cumsum(ctx)])

    def propose(seqs):
        n = len(seqs)
        sess = DflashSession(TINY, w, kv["page_table"][seqs], kv["n_pages"], block)
        rows = np.concatenate([np.arange(offs[b], offs[b + 1]) for b in seqs])
        sess.append(ctx[seqs], kv["k_rows"][:, rows], kv["v_rows"][:, rows])
        out = sess.block_buffers(with_logits=True)
        sess.propose(torch.from_numpy(anchors[seqs]).cuda(), 5, to_device_bf16(np.ascontiguousarray(feats[seqs])), 0.0,
                     None, out)
        torch.cuda.synchronize()
        assert int(sess.status.item()) == 0 and n == out["draft_tokens"].shape[0]
        return out["draft_tokens"].cpu().numpy(), out["draft_logits"].cpu().numpy()

    tok, z = propose(list(range(B)))
    for b in (0, 4, 8, 9):
        t1, z1 = propose([b])
        # the key ranges of the attention differ with a group's rows: float32 sums in another order, and a cached
        # bf16 row may round the other way (2^-8 of a key, attended with weight <= 1)
        assert np.abs(z[b] - z1[0]).max() < 2e-2
        gap = np.sort(z1[0], -1)
        sure = gap[:, -1] - gap[:, -2] > 4e-2
        assert (tok[b][sure] == t1[0][sure]).all()
