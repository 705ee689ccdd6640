"""FP64 grids on whole blocks of every width: with more grids than SMs two or four
narrower blocks share an SM, each with its part of the shared memory, and lines
are shared by fewer lanes.  What can go wrong sits where a grid's arrays move
between shared memory and the slice and where a class holds grids of several
sizes.  Node by node against the oracle, and prices of large batches against
the same instances alone (a block or a cluster per grid): 1e-12 of the largest
value, as the other FP64 paths.
"""
import numpy as np
import pytest

from launch_info import kernel_launches
from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from paper_2408_00559_gb300 import workloads as W
from test_gpu_parity import TOL64, check_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


@pytest.mark.parametrize("bc", ["neumann", "dirichlet"])
def test_one_problem_on_narrow_blocks(bc):
    # 2079 grids of 128 and 256 nodes, two blocks of 128 per SM
    import torch
    inst = dict(W.small_instance(6, 8, steps=1, seed=31), bc=bc)
    st = torch.cuda.Stream()
    prob = B.Problem(inst, stream=st)
    launched = kernel_launches(lambda: prob.step(1), st)
    sizes = prob.grid_info()[0].sum(axis=1)
    prob.close()
    assert any(b == 128 and g > torch.cuda.get_device_properties(0).multi_processor_count for g, b, _, _ in launched), launched
    big = [int(g) for g in np.flatnonzero(sizes == 8)]
    check_problem(inst, TOL64, TOL64, sample=big[:: len(big) // 6] + [int(np.flatnonzero(sizes == 7)[5])])


@pytest.mark.parametrize("N,level,full,count,bc", [
    (2, 4, True, 250, "neumann"), (2, 4, True, 500, "dirichlet"),   # 256 nodes: two, four blocks per SM
    (2, 5, True, 250, "neumann"), (2, 5, True, 500, "neumann"),     # 1024 nodes, factors in the slice
    (3, 3, True, 250, "dirichlet"), (3, 3, True, 500, "neumann"),   # 512 nodes
    (4, 2, True, 500, "neumann"), (8, 1, True, 500, "neumann"),
    (5, 2, True, 250, "neumann"), (2, 6, True, 250, "neumann"),     # 1024, 4096 nodes: two at most
    (2, 8, False, 40, "neumann"), (2, 10, False, 20, "dirichlet"),  # classes of several sizes, long lines
    (4, 7, False, 9, "neumann"),
])
def test_large_batches_price_like_single_problems(N, level, full, count, bc):
    import torch
    insts = [dict(W.small_instance(N, level, steps=2, seed=600 + s, full=full,
                                   payoff="caplet" if N == 2 else "swaption"), bc=bc) for s in range(count)]
    b = B.Batch(insts)
    out = torch.zeros(count, dtype=torch.float64, device="cuda")
    b.run(out.data_ptr())
    torch.cuda.synchronize()
    b.close()
    p = out.cpu().numpy()
    assert np.all(np.isfinite(p))
    for k in (0, count // 2, count - 1):
        prob = B.Problem(insts[k])
        prob.step(2)
        ref = prob.combine()
        scale = np.sum(np.abs(prob.grid_info()[1] * prob.grid_values())) * insts[k].get("discount", 1.0)
        prob.close()
        assert abs(p[k] - ref) <= TOL64 * scale, (k, p[k], ref)
