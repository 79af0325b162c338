"""The merge of the per-CTA lists where it can go wrong: scores that all tie (the bar cuts them
by index, also beyond 2^32), scores with many ties (exact integers, against the oracle), list
lengths around the 32-entry rows, and a range that leaves most lists empty."""
import numpy as np
import pytest

from paper_2609_02109_gb300 import workload as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_02109_gb300 import mf as m
    return m


@pytest.mark.parametrize("precision", ["fp32", "fp32_simt", "bf16"])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 100, 257, 1024])
def test_every_score_ties(mf, precision, k):
    prob = W.paper_scale()
    prob["obj_w"] = np.zeros(5, np.float32)
    prob["sla"] = np.full(5, 100.0, np.float32)
    if precision == "bf16" and k > 100:
        k = 100  # (the shortlist of 8 k has to fit the kernel's lists)
    with mf.Context(prob, precision=precision) as ctx:
        r = ctx.search(k)
        assert r["count"] == ctx.space_size
        assert (r["topk_score"] == 0.0).all()
        assert r["topk_idx"].tolist() == list(range(k))
        lo = ctx.space_size - 40  # a single tile: most lists stay empty
        r = ctx.search(k, lo=lo)
        assert r["topk_idx"].tolist()[:40] == list(range(lo, lo + 40))[:k]
        assert (r["topk_idx"][40:] == np.uint64(mf.EMPTY)).all() and np.isneginf(r["topk_score"][40:]).all()


@pytest.mark.parametrize("k", [3, 64, 300, 1024])
def test_many_ties_match_the_oracle(mf, oracle_mod, k):
    prob = W.integer_landscape([9, 7, 8, 6, 5], 21, 30.0)
    ti, ts, cnt = oracle_mod.Oracle(prob).exhaustive(k)
    assert len(np.unique(ts)) < k or k < 64  # the top holds ties
    with mf.Context(prob) as ctx:
        r = ctx.search(k)
    assert r["count"] == cnt
    assert np.array_equal(r["topk_idx"], ti) and np.array_equal(r["topk_score"].astype(np.float64), ts)


@pytest.mark.parametrize("k", [1, 5, 100, 1024])
@pytest.mark.parametrize("levels", [1, 3])
def test_ties_at_indices_beyond_2_32(mf, k, levels):
    """The last 300001 indices of 255^5: one score, or three that the last model's option
    chooses, spread over all lists."""
    prob = W.make_problem([255] * 5, 8, 32, 0, 34, 1e6, precision="fp32_simt")
    prob["obj_w"] = np.zeros(5, np.float32)
    prob["sla"] = np.full(5, 100.0, np.float32)
    prob["weights"][:] = 0.0
    if levels == 3:  # throughput of the last model = its first feature: 2, 1 or 0
        prob["obj_w"][4] = 1.0
        per = W.param_count(8, 32, 0)
        prob["local_feats"][4 * 255:, 0] = np.arange(255) % 3
        w = prob["weights"][4 * per:]
        w[0] = 1.0                 # W1[0, 0]
        w[32 * 12 + 32] = 1.0      # W3[0, 0]
    n = 255 ** 5
    lo = n - 300001
    idx = np.arange(lo, n, dtype=np.uint64)
    J = (idx % np.uint64(255) % np.uint64(3)).astype(np.float32) if levels == 3 else np.zeros(idx.size, np.float32)
    order = np.lexsort((idx, -J))[:k]
    with mf.Context(prob) as ctx:
        r = ctx.search(k, lo=lo, hi=n)
    assert r["count"] == 300001
    assert np.array_equal(r["topk_idx"], idx[order]) and np.array_equal(r["topk_score"], J[order])
