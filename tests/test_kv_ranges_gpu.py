"""K/V append in persistent blocks of 16-row groups: counts at the edges of a group, empty sequences between full ones,
more rows than one wave of blocks, more sequences than threads of a block, and a sequence whose page id is invalid."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from dataclasses import replace  # noqa: E402

from paper_2609_09338_gb300 import synthetic as syn  # noqa: E402
from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from parity import gather_positions  # noqa: E402
from test_kv_gpu import _built, _session  # noqa: E402,F401


@pytest.mark.parametrize("counts", [[0, 16, 0, 0, 17, 1, 0], [15], [33], [1] * 300 + [0] * 5, [5000, 0, 7001, 3]])
def test_rows_land_whatever_the_counts(counts):
    ctx = np.asarray(counts, np.int32)
    sess, kv = _session(replace(TINY, n_layers=2), ctx, 8, 21, spare=2)
    sess.append(ctx, kv["k_rows"], kv["v_rows"])
    torch.cuda.synchronize()
    assert int(sess.status.item()) == 0
    np.testing.assert_array_equal(sess.kv.seq_len.cpu().numpy(), ctx)
    pages = [p.view(torch.int16).cpu().numpy().view(np.uint16) for p in (sess.kv.k_pages, sess.kv.v_pages)]
    off = 0
    for b, n in enumerate(ctx):
        for got, want in zip(pages, (kv["k_rows"], kv["v_rows"])):
            np.testing.assert_array_equal(gather_positions(got, kv["page_table"][b], np.arange(n)), want[:, off:off + n])
        off += int(n)


def test_an_invalid_page_keeps_its_sequence_back():
    ctx = np.asarray([40, 20, 33], np.int32)
    sess, kv = _session(TINY, ctx, 8, 22)
    sess.kv.page_table[1, 1] = kv["n_pages"]
    sess.append(ctx, kv["k_rows"], kv["v_rows"])
    torch.cuda.synchronize()
    assert int(sess.status.item()) == -4
    np.testing.assert_array_equal(sess.kv.seq_len.cpu().numpy(), [40, 0, 33])
    got = gather_positions(sess.kv.k_pages.view(torch.int16).cpu().numpy().view(np.uint16), kv["page_table"][2],
                           np.arange(33))
    np.testing.assert_array_equal(got, kv["k_rows"][:, 60:93])
