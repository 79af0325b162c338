"""The fixed-context scan against numpy's float32 sums of the same table, bit for bit: the
counts by binary search and by two pointers, the bounds that settle whole settings, the bar
from the corner configurations and the slices cut at odd places."""
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


def brute(prob, ctx, k, lo, hi):
    """(count, top-k indices, scores) of [lo, hi): float32 sums in model order."""
    ks = [int(v) for v in prob["n_options"]]
    off = np.concatenate([[0], np.cumsum(ks)])
    _, _, u, ok = ctx.fc_table()
    idx = np.arange(lo, hi, dtype=np.uint64)
    J = np.zeros(idx.size, np.float32)
    V = np.zeros(idx.size, np.float32)
    good = np.ones(idx.size, bool)
    stride = 1
    digits = []
    for kk in reversed(ks):
        digits.append((idx // np.uint64(stride) % np.uint64(kk)).astype(np.int64))
        stride *= kk
    for i, d in enumerate(reversed(digits)):
        J = J + u[off[i] + d]
        V = V + np.asarray(prob["demand"], np.float32)[off[i] + d, 1]
        good &= ok[off[i] + d]
    good &= V <= np.float32(prob["vram_cap"])
    s, ix = J[good], idx[good]
    order = np.lexsort((ix, -s))[:k]
    return int(good.sum()), ix[order], s[order]


CASES = [  # options, cap, tau (None: as drawn)
    ([7], 9.0, None), ([255], 10.0, None), ([1, 1, 1], 50.0, None), ([2, 3], 12.0, None),
    ([40, 50], 20.0, -5.0), ([5, 6, 7, 8], 30.0, -5.0), ([5, 6, 7, 8], 42.0, None),
    ([23, 17, 21, 19], 40.0, -5.0),      # about half of the space fits
    ([23, 17, 21, 19], 14.0, -5.0),      # almost nothing fits: the corners hold few
    ([23, 17, 21, 19], 1.0, -5.0),       # nothing fits
    ([23, 17, 21, 19], 500.0, -5.0),     # everything fits
    ([9] * 6, 60.0, -5.0), ([2] * 16, 150.0, -5.0), ([30, 29, 31, 28], 40.0, -5.0),
]


@pytest.mark.parametrize("options,cap,tau", CASES)
@pytest.mark.parametrize("k", [1, 32, 64, 65, 1000])
def test_scan_is_the_brute_force(mf, options, cap, tau, k):
    prob = W.make_problem(options, 8, 32, 0, 40 + len(options), cap)
    fc = W.fc_scenario(prob, 40 + len(options))
    if tau is not None:
        fc["tau"] = np.full(len(options), tau, np.float32)
    with mf.Context(prob) as ctx:
        ctx.fc_set(fc)
        total = ctx.space_size
        ranges = [(0, total, 0), (total // 3, total - total // 7, 0), (total // 2, min(total, total // 2 + 3), 0),
                  (0, total, total // 5 + 1)]
        for lo, hi, chunk in ranges:
            count, ti, ts = brute(prob, ctx, k, lo, hi)
            r = ctx.fc_search(k, lo=lo, hi=hi, chunk=chunk)
            assert r["count"] == count
            n = ti.size
            assert np.array_equal(r["topk_idx"][:n], ti) and np.array_equal(r["topk_score"][:n], ts)
            assert (r["topk_idx"][n:] == np.uint64(mf.EMPTY)).all()


@pytest.mark.parametrize("special", ["cap_on_a_sum", "equal_terms", "inf_demand", "nan_demand", "inf_quality",
                                     "plus_inf_demand", "inf_cap", "inf_cap_and_demand", "minus_inf_cap", "large_demands"])
def test_special_values(mf, special):
    options = [11, 12, 13]
    prob = W.make_problem(options, 8, 32, 0, 77, 30.0)
    dem = prob["demand"]
    fc = W.fc_scenario(prob, 77)
    fc["tau"] = np.full(3, 0.1 if "inf_cap" in special else -5.0, np.float32)  # (0.1: some options below)
    if special == "cap_on_a_sum":  # the bound is inclusive
        prob["vram_cap"] = float((dem[3, 1] + dem[11 + 5, 1]) + dem[23 + 7, 1])
    elif special == "equal_terms":
        fc["quality"] = np.zeros(36, np.float32)
        fc["beta"], fc["alpha"] = 0.0, 0.0
        dem[:, 1] = 4.0
    elif special == "inf_demand":
        dem[[2, 15, 30], 1] = [np.inf, -np.inf, np.inf]
    elif special == "plus_inf_demand":
        dem[[2, 15, 30], 1] = np.inf
    elif special.startswith("inf_cap") or special == "minus_inf_cap":
        prob["vram_cap"] = -np.inf if special == "minus_inf_cap" else np.inf
        if special == "inf_cap_and_demand":
            dem[[2, 15, 30], 1] = np.inf
    elif special == "large_demands":  # sums beyond fp32's range, of either sign
        dem[:, 1] *= np.float32(1e37)
        dem[11:17, 1] *= -1
    elif special == "nan_demand":
        dem[[0, 20], 1] = np.nan
    else:
        fc["quality"][[4, 17]] = np.inf
    with mf.Context(prob) as ctx:
        ctx.fc_set(fc)
        with np.errstate(invalid="ignore", over="ignore"):
            count, ti, ts = brute(prob, ctx, 40, 0, ctx.space_size)
        assert "inf_cap" not in special or not ctx.fc_table()[3].all()
        r = ctx.fc_search(40)
        assert r["count"] == count
        if special != "inf_quality":
            assert np.array_equal(r["topk_idx"][:ti.size], ti) and np.array_equal(r["topk_score"][:ts.size], ts)


@pytest.mark.parametrize("k", [5, 100])
def test_corner_values_that_overflow(mf, k):
    """Demands next to each other near fp32's end and utilities of order 1e34: the corner's
    J - lambda V overflows for options that meet their floors, between others that do not."""
    options = [12, 13]
    prob = W.make_problem(options, 8, 32, 0, 91, 3e38)
    prob["demand"][:, 1] = np.float32(1e38) * (1 + np.arange(25, dtype=np.float32) % 11 * np.float32(2.0 ** -23))
    fc = W.fc_scenario(prob, 91)
    fc["omega"] = np.full(2, 1e34, np.float32)
    fc["tau"] = np.full(2, -5.0, np.float32)
    with mf.Context(prob) as ctx:
        ctx.fc_set(fc)
        f = ctx.fc_table()[1]
        fc["tau"] = np.array([np.sort(f[:12])[5], np.sort(f[12:])[6]], np.float32)
        ctx.fc_set(fc)
        count, ti, ts = brute(prob, ctx, k, 0, ctx.space_size)
        r = ctx.fc_search(k)
        assert count == 7 * 7 and r["count"] == count
        assert np.array_equal(r["topk_idx"][:ti.size], ti) and np.array_equal(r["topk_score"][:ts.size], ts)


@pytest.mark.parametrize("k", [1, 32, 64, 65, 300])
@pytest.mark.parametrize("levels", ["one", "few"])
@pytest.mark.parametrize("cap", [500.0, 52.0])
def test_equal_scores(mf, k, levels, cap):
    """Utilities of one value, or of a reload cost paid or not: by index among equals, where
    whole settings of the leading models only tie with the bar."""
    options = [24, 23, 22, 21, 5]
    prob = W.make_problem(options, 8, 32, 0, 93, cap)
    fc = W.fc_scenario(prob, 93)
    fc["tau"] = np.full(5, -5.0, np.float32)
    fc["omega"] = np.zeros(5, np.float32)
    fc["prev_variant"] = np.zeros(5, np.int32)
    fc["beta"], fc["alpha"] = 0.0, 0.0 if levels == "one" else 1.0 / 60.0
    with mf.Context(prob) as ctx:
        ctx.fc_set(fc)
        total = ctx.space_size
        for lo, hi in ((0, total), (total // 3, total - 7)):
            count, ti, ts = brute(prob, ctx, k, lo, hi)
            r = ctx.fc_search(k, lo=lo, hi=hi)
            assert r["count"] == count
            assert np.array_equal(r["topk_idx"], ti) and np.array_equal(r["topk_score"], ts)
