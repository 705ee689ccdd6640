"""The autotuner's choice between shared and global memory, class by class, in a
batch that has both kinds: a class that is moved changes the order of a solve's
launches, so times are compared by class.

The batch: d=4 level-7 mixed-precision instances, whose grids of 128 nodes run
on whole blocks and take several times longer with their state in global
memory, and one tiny instance whose grids are forced there and take next to no
time.  The first class must stay where it is.
"""
import pytest

from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from paper_2408_00559_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


def run_ms(b, out):
    import torch
    t = []
    for _ in range(4):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        b.run(out.data_ptr())
        e1.record()
        torch.cuda.synchronize()
        t.append(e0.elapsed_time(e1))
    return min(t[1:])


def test_placement_is_chosen_by_the_class_own_times():
    import torch
    insts = [W.small_instance(4, 7, steps=8, seed=s, precision="mixed") for s in range(40)]
    insts.append(dict(W.small_instance(4, 1, steps=8, seed=99, precision="mixed"), global_grids=True))
    b = B.Batch(insts)
    b.set_kappa_max(0)
    before = b.classes()
    assert before[1] == 1 and before[2] == 1, before
    out = torch.zeros(len(insts), dtype=torch.float64, device="cuda")
    t0 = run_ms(b, out)
    b.autotune(3)
    t1 = run_ms(b, out)
    assert b.classes() == before, (before, b.classes(), t0, t1)
    b.close()
