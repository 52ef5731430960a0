"""The pick of a draft token from the LM head's 32-id partials: vocabularies of one group, of fewer groups than warps, of
a partial last group, and of more partials than a lane holds (read again from memory), greedy and sampled, with one and
with several candidates, against the oracle and the call's own logits."""
from dataclasses import replace

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import drafter as od  # noqa: E402
from paper_2609_09338_gb300.workloads import TINY  # noqa: E402
from test_draft_gpu import _built, check_case, run_case  # noqa: E402,F401
from test_tree_gpu import _draft_topk  # noqa: E402


@pytest.mark.parametrize("V,T", [(20, 0.0), (33, 1.0), (1000, 1.0), (32773, 0.0), (32773, 1.0), (270001, 0.0), (270001, 1.0)])
def test_one_candidate(V, T):
    check_case(run_case(replace(TINY, vocab=V), [3, 17, 40, 9], 3, T, 60 + V % 7, peaked=T > 0))


@pytest.mark.parametrize("V,k,T", [(33, 8, 0.0), (5000, 5, 0.0), (270001, 8, 0.0), (270001, 3, 1.0), (64, 8, 1.0)])
def test_several_candidates(V, k, T):
    res, inp = _draft_topk(replace(TINY, vocab=V), [4, 30, 12], 3, k, T, 77, peaked=T > 0)
    tr = res["tree"]
    assert tr["status"] == 0
    np.testing.assert_array_equal(tr["cand"][..., 0], res["chain"]["draft_tokens"])
    z = tr["draft_logits"].astype(np.float64)
    for b in range(z.shape[0]):
        for i in range(z.shape[1]):
            if T == 0:
                order = np.lexsort((np.arange(V), -z[b, i]))[:k + 1]
                # recomputed in another order: ranks are sure where neighbours are 1e-4 apart
                gaps = -np.diff(z[b, i][order])
                for j in range(1, min(k, V)):
                    if gaps[j - 1] > 1e-4 and (j >= len(gaps) or gaps[j] > 1e-4):
                        assert tr["cand"][b, i, j] == order[j], (b, i, j)
            else:
                for j in range(k):
                    own = od.sample(z[b, i], T, float(inp["u"][b, i, j]))
                    if own["margin"] > 1e-5:
                        assert tr["cand"][b, i, j] == own["token"], (b, i, j)
