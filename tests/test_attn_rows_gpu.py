"""Attention of a sequence's extend rows in tiles of 16 (row, head) queries: every group size and head width, tiles that
are partly filled, several tiles a sequence, key ranges that end inside a page or before a split, against the oracle."""
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from test_draft_gpu import _built, check_case, run_case  # noqa: E402,F401


@pytest.mark.parametrize("heads,kv_heads,hd,max_new,ctx", [
    (4, 4, 64, 10, [0, 1, 15, 16, 40, 17, 31, 2]),
    (16, 8, 64, 9, [130, 5, 64, 0, 33]),
    (32, 8, 128, 10, [1100, 3, 47, 2200]),
    (32, 4, 128, 20, [31, 16, 1025, 90]),
    (4, 4, 128, 64, [20, 300, 0]),
])   # rows x KV heads above 304: fewer run on the decode kernel
def test_extend_rows_share_their_keys(heads, kv_heads, hd, max_new, ctx):
    shape = replace(TINY, n_q_heads=heads, n_kv_heads=kv_heads, head_dim=hd, n_layers=2)
    rng = np.random.default_rng(heads + hd)
    n_new = rng.integers(1, max_new + 1, size=len(ctx))
    n_new[0] = max_new
    check_case(run_case(shape, ctx, 2, 0.0, 90 + heads + hd, n_new=n_new, max_new=max_new))
