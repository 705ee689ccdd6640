"""The launches of a step that are forked off the caller's stream keep the
caller's stream priority (a problem with warp groups and whole blocks, on a
stream of the highest priority and on one of the default)."""
import pytest

from launch_info import kernel_launches
from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from paper_2408_00559_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("high", [True, False])
def test_forked_launches_keep_the_priority(high):
    import torch
    BLD.build()
    st = torch.cuda.Stream(priority=-1 if high else 0)
    prob = B.Problem(W.small_instance(4, 7, steps=2, seed=5), stream=st)
    launched = kernel_launches(lambda: prob.step(1), st)
    prob.close()
    assert len(launched) >= 2, launched
    assert {p for _, _, _, p in launched} == {st.priority}, (launched, st.priority)
