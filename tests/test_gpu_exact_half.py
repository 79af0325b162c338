"""The exact tensor-core variant where its operands' ranges are put to the test: features,
weights and demands far from order one, zero columns and units, an outlier option, every
model count (one to three weight passes), the longest lists.  1e-5 of the oracle everywhere."""
import numpy as np
import pytest

from paper_2609_02109_gb300 import workload as W
from _parity import check_scores

pytestmark = pytest.mark.gpu

DL, H, DIN = 8, 64, 12
PER = W.param_count(DL, H, H)


@pytest.fixture(scope="module")
def mf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_02109_gb300 import mf as m
    return m


def _views(prob, i):
    w = prob["weights"][i * PER:(i + 1) * PER]
    return w[:H * DIN].reshape(H, DIN), w[H * DIN:H * DIN + H], w[H * DIN + H:H * DIN + H + H * H].reshape(H, H)


def _vary(prob, what):
    n = len(prob["n_options"])
    off = np.concatenate([[0], np.cumsum(prob["n_options"])])
    for i in range(n):
        w1, b1, w2 = _views(prob, i)
        x = prob["local_feats"][off[i]:off[i + 1]]
        if what == "large_features":      # x 2^20, their weights down by as much
            x *= np.float32(2.0 ** 20)
            w1[:, :DL] *= np.float32(2.0 ** -20)
        elif what == "small_features":
            x *= np.float32(1e-9)
            w1[:, :DL] *= np.float32(1e9)
        elif what == "one_large_column":
            x[:, 3] *= np.float32(3e4)
            w1[:, 3] *= np.float32(1.0 / 3e4)
        elif what == "zeros":
            x[:, 1] = 0.0
            w1[7] = 0.0
            b1[7] = 0.0
            w2[9] = 0.0
        elif what == "large_units":       # hidden units far apart, made up for in the next layer
            s = np.float32(2.0) ** np.arange(-16, 16, 0.5).astype(np.int32).astype(np.float32)
            w1 *= s[:, None]
            b1 *= s
            w2 /= s[None, :]
        elif what == "outlier":
            x[0] *= np.float32(1e6)
        elif what == "no_aggregate":
            w1[:, DL:] = 0.0
    return prob


@pytest.mark.parametrize("what", ["plain", "large_features", "small_features", "one_large_column", "zeros", "large_units",
                                  "outlier", "no_aggregate", "sigmoid"])
def test_ranges(mf, oracle_mod, what):
    import torch
    prob = W.make_problem([9, 8, 7, 6], DL, H, H, 31, 45.0, objective="soft_lat", soft_penalty=0.1,
                          out_act="sigmoid" if what == "sigmoid" else "identity")
    _vary(prob, what)
    o = oracle_mod.Oracle(prob)
    idx = np.arange(o.space_size(), dtype=np.uint64)
    rs, rf, rp, ra = o.score_list(idx, with_pred=True)
    with mf.Context(prob) as ctx:
        assert ctx.stats()["scoring_path"] == 2
        s, f, p = (t.cpu().numpy() for t in ctx.score_batch(torch.from_numpy(idx.astype(np.int64)).cuda(), with_pred=True))
        r = ctx.search(64)
    check_scores(prob, s, f, rs, rf, rp, ra, got_pred=p)
    order = np.lexsort((idx[f > 0], -s[f > 0]))[:64]
    assert np.array_equal(r["topk_idx"], idx[f > 0][order]) and r["count"] == int((f > 0).sum())


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("k", [5, 1024])
def test_model_counts_and_long_lists(mf, n, k):
    import torch
    prob = W.make_problem([7, 5, 6, 4, 5, 3, 4, 3][:n], DL, H, H, 50 + n, 11.0 * n)
    with mf.Context(prob) as ctx, mf.Context(prob, precision="fp32_simt") as ref:
        a, b = ctx.search(k), ref.search(k)
        assert a["count"] == b["count"]
        fin = np.isfinite(b["topk_score"])
        assert np.array_equal(np.isfinite(a["topk_score"]), fin)
        assert np.allclose(a["topk_score"][fin], b["topk_score"][fin], rtol=0, atol=1e-5 * max(1.0, np.abs(b["topk_score"][fin]).max(initial=0.0)))
        # a list scores the same numbers, but for the order of the N terms' sum: models run in
        # weight passes, whose partial sums round apart (at most N ulps of N terms of order
        # one: 8 * 8 * 2^-24)
        sa, _ = ctx.score_batch(torch.from_numpy(a["topk_idx"][fin].astype(np.int64)).cuda())
        assert np.abs(sa.cpu().numpy() - a["topk_score"][fin]).max(initial=0.0) <= 64 * 2.0 ** -24
