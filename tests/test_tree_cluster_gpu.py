"""Tree verification at the edges of its split over a cluster of 1 to 8 blocks in chunks of 256 ids: vocabularies smaller
than a chunk, one past a whole number of chunks, unaligned rows, slices that do not fit shared memory (later passes read
the rows again), every cluster size (tree_cluster of csrc/sizes.h), and more sequences than one wave."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import tree as ot  # noqa: E402
from paper_2609_09338_gb300 import synthetic as syn  # noqa: E402
from test_tree_gpu import RATIO_BAND, _built, _run_tree, check_tree  # noqa: E402,F401


@pytest.mark.parametrize("V,B,K,k,T,dtype", [
    (40, 6, 3, 2, 1.0, "f32"), (257, 6, 3, 3, 1.0, "f32"), (2056, 6, 2, 8, 0.7, "bf16"), (1001, 6, 3, 2, 0.7, "bf16"),
    (300, 5, 3, 2, 0.0, "f32"), (2049, 5, 2, 2, 0.0, "bf16"), (262152, 2, 2, 2, 1.0, "f32"),
    (262151, 2, 2, 2, 1.0, "f32"),
    (4096, 3, 2, 3, 1.0, "f32"), (4099, 3, 2, 3, 0.7, "f32"), (16000, 3, 2, 3, 1.0, "bf16"), (9001, 3, 2, 3, 1.0, "f32"),
    (30001, 3, 2, 3, 1.0, "f32"), (50304, 3, 2, 3, 0.0, "bf16"), (3001, 310, 1, 2, 1.0, "f32"), (30008, 160, 1, 2, 1.0, "f32"),
    (3008, 470, 1, 2, 0.0, "bf16"), (3001, 470, 1, 2, 0.0, "f32"),
])
def test_tree_walk_over_a_cluster(V, B, K, k, T, dtype):
    ti = syn.make_tree_inputs(V, B, K, k, T, 0.7, seed=V + B + k)
    g = _run_tree(ti, T, dtype)
    assert g["status"] == 0
    conv = (lambda a: a) if dtype == "f32" else syn.bf16_bits
    o = ot.verify_tree(conv(ti["target_logits"]), conv(ti["draft_logits"]) if T > 0 else None, ti["cand"], T,
                       ti["u_accept"], ti["u_sample"], ratio_band=RATIO_BAND)
    assert check_tree(g, o, K) <= max(1, B // 4)
