"""Block drafting keeps one order of summation.

Mask positions leave much of the draft mass on ids of 1e-6 beside a leading one.  A float32 drafter's leading logit is
some 1e-5 off, which moves the cumulative sum past several such ids, so any other order of any sum on the way draws
neighbouring ids.  The ids and logits of a call are the same bit for bit whatever else is drafted in it, and the ids are
those recorded in tests/golden/block_ids.json.
"""
import json
import os
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle.bf16 import widen  # noqa: E402
from paper_2609_09338_gb300 import synthetic as syn  # noqa: E402
from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from test_dflash_gpu import _built  # noqa: E402,F401

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "block_ids.json")
# groups of 5 + 3 and of 8 + 1 sequences (the last one with one LM-head segment)
CASES = {
    "d512-b8-blk16": (replace(TINY, d_model=512, n_layers=4, n_q_heads=8, n_kv_heads=2, ffn_dim=4096, feat_dim=4096,
                              vocab=262144), [30, 1, 64, 17, 5, 90, 200, 41], 16),
    "d1024-b9-blk11": (replace(TINY, d_model=1024, n_layers=2, n_q_heads=8, n_kv_heads=4, ffn_dim=2048, feat_dim=4096,
                               vocab=131072), [700, 3, 9, 61, 2, 18, 33, 150, 40], 11),
}


def make(shape, ctx, block, seed):
    """Weights whose head gives each token one successor of about half the mass, and a call's inputs."""
    w = syn.make_weights(shape, seed)
    rng = np.random.default_rng(seed + 1)
    embed = widen(w["embed"]) * np.float32(50)                      # N(0, 1)
    w["embed"] = syn.bf16_bits(embed)
    gain = np.log(shape.vocab) * np.sqrt(1 + shape.n_layers * shape.d_model / 2560) / shape.d_model
    w["lm_head"] = syn.bf16_bits(widen(w["lm_head"]) + np.float32(gain) * embed[rng.permutation(shape.vocab)])
    B, P = len(ctx), block - 1
    return {"shape": shape, "block": block, "ctx": np.asarray(ctx, np.int32), "w": w,
            "kv": syn.make_kv_prefix(shape, np.asarray(ctx, np.int32), P, seed + 2),
            "anchors": rng.integers(0, shape.vocab, size=B).astype(np.int32),
            "feats": syn.make_draft_inputs(shape, B, 1, 1, seed + 3)["feats"][:, 0],
            "u": rng.random((B, P), dtype=np.float32)}


def propose(c, T, seqs=None, refused=()):
    from paper_2609_09338_gb300.binding import to_device_bf16
    from paper_2609_09338_gb300.session import DflashSession
    seqs = list(range(len(c["ctx"]))) if seqs is None else seqs
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    offs = np.concatenate([[0], np.cumsum(c["ctx"])])
    rows = np.concatenate([np.arange(offs[b], offs[b + 1]) for b in seqs])
    kv = c["kv"]
    sess = DflashSession(c["shape"], c["w"], kv["page_table"][seqs], kv["n_pages"], c["block"])
    sess.append(c["ctx"][seqs], kv["k_rows"][:, rows], kv["v_rows"][:, rows])
    for b in refused:                # pages outside the pool: the call reports and skips these sequences
        sess.kv.page_table[b] = -1
    out = sess.block_buffers(with_logits=True)
    sess.propose(dev(c["anchors"][seqs]), 5, to_device_bf16(np.ascontiguousarray(c["feats"][seqs])), T,
                 dev(c["u"][seqs]), out)
    torch.cuda.synchronize()
    assert (int(sess.status.item()) != 0) == bool(refused)
    return {k: v.cpu().numpy() for k, v in out.items()}


def ids_of(name):
    shape, ctx, block = CASES[name]
    return propose(make(shape, ctx, block, 91), 1.0)


@pytest.mark.parametrize("name", sorted(CASES))
def test_sampled_ids_are_the_recorded_ones(name):
    with open(GOLDEN) as f:
        want = np.array(json.load(f)[name], np.int32)
    np.testing.assert_array_equal(ids_of(name)["draft_tokens"], want)


@pytest.mark.parametrize("block,T", [(16, 1.0), (11, 0.0), (24, 1.0)])
def test_groups_do_not_change_one_another(block, T):
    """A call's groups of up to 80 rows give bit for bit what each gives in a call of its own."""
    shape = replace(TINY, d_model=768, n_layers=2, n_q_heads=4, vocab=32768)
    P = block - 1
    B, group = 2 * (80 // P) + 1, 80 // P
    c = make(shape, np.random.default_rng(block).integers(1, 200, size=B), block, 71)
    whole = propose(c, T)
    for b0 in range(0, B, group):
        seqs = list(range(b0, min(B, b0 + group)))
        own = propose(c, T, seqs)
        for k in own:
            np.testing.assert_array_equal(whole[k][seqs], own[k], err_msg=f"{k} of group {b0}")


@pytest.mark.parametrize("refused", [range(5, 10), range(0, 5), range(5, 13)])
def test_a_refused_group_leaves_the_others(refused):
    """Attention runs once a group: one without a valid row ends early, and what follows still waits for the others."""
    shape = replace(TINY, n_layers=3, ffn_dim=4096)
    c = make(shape, np.random.default_rng(4).integers(1, 900, size=13), 16, 23)
    whole, some = propose(c, 1.0), propose(c, 1.0, refused=refused)
    kept = [b for b in range(13) if b not in refused]
    for k in whole:
        np.testing.assert_array_equal(some[k][kept], whole[k][kept], err_msg=k)
    assert (some["draft_tokens"][list(refused)] == -1).all()


@pytest.mark.parametrize("B,block", [(63, 16), (66, 16), (160, 4), (13, 65)])
def test_passes_do_not_change_one_another(B, block):
    """Calls of more than 512 rows run in several passes over one workspace, the last one smaller: every group's results
    are those of a call of its own."""
    P = block - 1
    group = 80 // P
    full = 512 // P // group * group
    assert B > full and B % full, "a smaller last pass"
    c = make(TINY, np.random.default_rng(B).integers(1, 60, size=B), block, 17)
    whole = propose(c, 1.0)
    last = (B - 1) // group * group
    for b0 in {0, full - group, (B // full) * full, last}:
        seqs = list(range(b0, min(B, b0 + group)))
        own = propose(c, 1.0, seqs)
        for k in own:
            np.testing.assert_array_equal(whole[k][seqs], own[k], err_msg=f"{k} of group {b0}")


def test_workspaces_grow_with_the_batch():
    """A workspace made for some batch is enough for every smaller one."""
    from paper_2609_09338_gb300 import binding as ob
    for shape in (TINY, replace(TINY, d_model=1024, n_q_heads=8, ffn_dim=4096, feat_dim=3072)):
        ctx = ob.osprey_create(shape, ob.upload_weights(syn.make_weights(shape, 5)))
        for max_new, max_pages in ((1, 4), (3, 40), (8, 300)):
            sizes = [ob.osprey_draft_workspace_bytes(ctx, B, 4, max_new, max_pages) for B in [*range(1, 700), 4095, 4097]]
            assert sizes == sorted(sizes), (max_new, max_pages)
        for block in (4, 16, 24, 81):
            sizes = [ob.osprey_dflash_workspace_bytes(ctx, B, block, 40) for B in range(1, 200)]
            assert sizes == sorted(sizes), block
