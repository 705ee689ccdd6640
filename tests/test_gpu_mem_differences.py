"""FP64 grids with their state in global memory, with and without stored
central differences: a batch whose vectors exceed the L2 cache evaluates the
stencil directly, the same instances alone from differences.  Both forms take
the same differences of the same values: 1e-12 of the largest value, as the
other FP64 paths."""
import numpy as np
import pytest

from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from paper_2408_00559_gb300 import workloads as W
from test_gpu_parity import TOL64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


@pytest.mark.parametrize("N,level,count,bc", [(4, 4, 64, "neumann"), (4, 4, 64, "dirichlet"), (3, 6, 40, "neumann"),
                                              (6, 3, 24, "neumann"), (2, 7, 24, "neumann")])
def test_direct_stencil_prices_like_stored_differences(N, level, count, bc):
    import torch
    insts = [dict(W.small_instance(N, level, steps=2, seed=800 + s, full=True, payoff="caplet" if N == 2 else "swaption"),
                  bc=bc) for s in range(count)]
    b = B.Batch(insts)
    assert b.classes()[2] == 1
    out = torch.zeros(count, dtype=torch.float64, device="cuda")
    b.run(out.data_ptr())
    torch.cuda.synchronize()
    b.close()
    p = out.cpu().numpy()
    for k in (0, count // 2, count - 1):
        prob = B.Problem(insts[k])
        prob.step(2)
        ref = prob.combine()
        prob.close()
        assert abs(p[k] - ref) <= TOL64 * abs(ref), (k, p[k], ref)
