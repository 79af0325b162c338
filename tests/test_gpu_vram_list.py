"""The VRAM-feasible index list at its edges: option counts of the last model around the lanes
a warp gives a setting, ranges cut inside a setting, bounded buffers, non-finite demands."""
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


@pytest.mark.parametrize("options,cap", [
    ([9], 10.0), ([255], 10.0), ([40, 1], 9.0), ([61, 47, 2], 30.0), ([31, 29, 3], 32.0), ([13, 17, 19, 31], 40.0),
    ([13, 17, 19, 32], 44.0), ([13, 17, 19, 33], 44.0), ([5, 6, 70], 33.0), ([40, 255], 20.0), ([2] * 14, 147.0),
    ([70, 70, 70], 4.0), ([70, 70, 70], 1000.0),
    # either side of the line between the counting kernels, segments of one and two steps
    ([13, 17, 4, 31], 40.0), ([13, 17, 5, 31], 40.0), ([40, 40, 40, 8, 3], 50.0), ([40, 40, 40, 9, 3], 50.0),
    ([255, 255, 3], 30.0), ([3, 140, 129], 30.0),
])
@pytest.mark.parametrize("special", [None, "nonfinite"])
def test_list_is_the_brute_force(mf, options, cap, special):
    prob = W.make_problem(options, 8, 32, 0, 60 + len(options), cap)
    if special:
        prob["demand"][[0, -1], 1] = [np.nan, -np.inf]
    off = np.concatenate([[0], np.cumsum(options)])
    V = np.zeros(1, np.float32)
    with np.errstate(invalid="ignore"):
        for i, k in enumerate(options):
            V = (V[:, None] + prob["demand"][off[i]:off[i] + k, 1][None, :].astype(np.float32)).reshape(-1)
        want = np.flatnonzero(V <= np.float32(cap))
    total = V.size
    with mf.Context(prob) as ctx:
        for lo, hi in ((0, total), (total // 3 + 1, total - total // 5), (total // 2, total // 2 + 1), (0, 0)):
            here = want[(want >= lo) & (want < hi)]
            for buf in (None, here.size // 2 + 1, 0):
                n, idx = ctx.vram_feasible(lo, hi, cap=buf)
                assert n == here.size
                keep = here if buf is None else here[:buf]
                assert np.array_equal(idx.cpu().numpy(), keep)
