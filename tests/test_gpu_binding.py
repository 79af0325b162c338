"""The binding around the C ABI: closed contexts, the current stream."""
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


def test_a_closed_context_is_refused(mf):
    prob = W.make_problem([5, 4], 8, 32, 0, 3, 40.0)
    with mf.Context(prob) as ctx:
        assert ctx.space_size == 20
    for call in (lambda: ctx.space_size, lambda: ctx.search(4), lambda: ctx.search(4, 0, 20),
                 lambda: ctx.fc_search(4), lambda: ctx.vram_feasible()):
        with pytest.raises(mf.MFError) as e:
            call()
        assert e.value.status == mf.MF_EINVAL


@pytest.mark.parametrize("raw", [True, False])
def test_calls_run_on_the_current_stream(mf, monkeypatch, raw):
    """With torch's raw stream query and, where a torch has none, with its public one."""
    import torch
    if not raw:
        monkeypatch.setattr(mf, "_raw_stream", None)
    prob = W.make_problem([9, 8, 7], 8, 64, 64, 3, 40.0)
    idx = torch.arange(504, dtype=torch.int64, device="cuda")
    with mf.Context(prob) as ctx:
        want = ctx.search(8)
        assert mf._stream(ctx.device) == torch.cuda.current_stream().cuda_stream
        torch.cuda.synchronize()
        with torch.cuda.stream(torch.cuda.Stream()) as _:
            st = torch.cuda.current_stream()
            assert mf._stream(ctx.device) == mf._stream(idx.device) == st.cuda_stream != 0
            got = ctx.search(8)
            score, _ = ctx.score_batch(idx)
            st.synchronize()
        assert np.array_equal(got["topk_idx"], want["topk_idx"]) and np.array_equal(got["topk_score"], want["topk_score"])
        assert np.array_equal(score.cpu().numpy()[want["topk_idx"].astype(np.int64)], want["topk_score"])
