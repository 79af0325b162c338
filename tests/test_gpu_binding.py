"""The binding around the C ABI: closed contexts."""
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
