"""Attention of a sequence's extend rows in tiles of 16 (row, head) queries: every group size and head width, tiles that
are partly filled, several tiles a sequence, key ranges that end inside a page or before a split, one range and many,
against the oracle.  The page tables are wide (``keys``), which is what takes small contexts to this kernel."""
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2609_09338_gb300 import synthetic as syn  # noqa: E402
from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from test_draft_gpu import _built, check_case, run_case  # noqa: E402,F401


@pytest.fixture
def wide_tables(monkeypatch):
    """Page tables padded to a number of keys; no sequence reaches the added pages."""
    made = syn.make_kv_prefix

    def pad_to(keys):
        def make(*args, **kw):
            kv = made(*args, **kw)
            more = keys // 16 - kv["page_table"].shape[1]
            assert more >= 0
            kv["page_table"] = np.pad(kv["page_table"], ((0, 0), (0, more)), mode="edge")
            return kv
        monkeypatch.setattr(syn, "make_kv_prefix", make)
    return pad_to


def pays(shape, B, max_new, keys):   # attn_rows_pays of csrc/sizes.h
    G = shape.n_q_heads // shape.n_kv_heads
    return max_new > 1 and max_new * G >= 8 and B * max_new * shape.n_kv_heads * (G + 2) * keys >= 6000000


@pytest.mark.parametrize("heads,kv_heads,hd,max_new,ctx,keys", [
    (4, 4, 64, 10, [0, 1, 15, 16, 40, 17, 31, 2], 8192),
    (16, 8, 64, 9, [130, 5, 64, 0, 33], 4608),
    (32, 8, 128, 10, [1100, 3, 47, 2200], 4096),
    (32, 4, 128, 20, [31, 16, 1025, 90], 2048),
    (4, 4, 128, 64, [20, 300, 0], 16384),
    (8, 8, 64, 8, list(range(0, 400, 5)), 512),   # one key range
])
def test_extend_rows_share_their_keys(wide_tables, heads, kv_heads, hd, max_new, ctx, keys):
    shape = replace(TINY, n_q_heads=heads, n_kv_heads=kv_heads, head_dim=hd, n_layers=2)
    assert pays(shape, len(ctx), max_new, keys)
    wide_tables(keys)
    rng = np.random.default_rng(heads + hd)
    n_new = rng.integers(1, max_new + 1, size=len(ctx))
    n_new[0] = max_new
    seqs = None if len(ctx) < 16 else [0, 7, 41, len(ctx) - 1]
    check_case(run_case(shape, ctx, 2, 0.0, 90 + heads + hd, n_new=n_new, max_new=max_new, sample_seqs=seqs))
