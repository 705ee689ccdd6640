"""FP64 grids on clusters whose right-hand sides do not fit in shared memory.

With 8192 Inner nodes three vectors of a grid fit in a block's shared memory
and the fourth, the right-hand side, lies in the cluster's slice of global
scratch.  Lines along the split axis then read it from there, and every later
axis's values from the owners' shared memory.  The problems below have such
grids whose longest axis, the split one, is the first that is solved (a rate),
is a later rate and is V, under both boundary conditions, on clusters of four
and eight blocks.  The bound is that of the other FP64 paths (1e-12 of the
largest value of a grid, node by node).
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


def instance(N, level, psi, bc):
    inst = W.small_instance(N, level, psi=psi, steps=2, seed=4000 + 10 * N + psi,
                            payoff="caplet" if N == 2 else "swaption")
    return dict(inst, bc=bc)


CASES = [
    # (N, level, psi, grids in shared memory, blocks of a cluster)
    (2, 9, 2, 15, 4),   # nine of 4096 nodes, six of 8192, (7, 6) and (6, 7) among them
    (3, 1, 4, 4, 8),    # (5, 4, 4), (4, 5, 4), (4, 4, 5) and (4, 4, 4)
    (4, 1, 3, 5, 8),    # (4, 3, 3, 3) and its kin
    (6, 1, 2, 2, 4),    # (3, 2, 2, 2, 2, 2) on four blocks of two rows
]
IDS = [f"N{c[0]}_n{c[1]}_psi{c[2]}" for c in CASES]


@pytest.mark.parametrize("bc", ["neumann", "dirichlet"])
@pytest.mark.parametrize("case", CASES, ids=IDS)
def test_right_hand_sides_in_the_slice_match_oracle(case, bc):
    import torch
    N, level, psi, grids, csize = case
    inst = instance(N, level, psi, bc)
    st = torch.cuda.Stream()
    prob = B.Problem(inst, stream=st)
    launched = kernel_launches(lambda: prob.step(1), st)
    prob.close()
    assert any(c == csize and g == csize * grids for g, _, c, _ in launched), launched
    check_problem(inst, TOL64, TOL64)


@pytest.mark.parametrize("case", CASES, ids=IDS)
def test_noalloc_prices_the_same(case):
    import torch
    N, level, psi, _, _ = case
    inst = instance(N, level, psi, "neumann")
    prob = B.Problem(inst)
    prob.step(inst["n_steps"])
    ref = prob.combine()
    scale = np.sum(np.abs(prob.grid_info()[1] * prob.grid_values())) * inst.get("discount", 1.0)
    prob.close()
    out = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    B.solve_noalloc([inst], out.data_ptr())
    torch.cuda.synchronize()
    assert abs(out.item() - ref) <= TOL64 * scale, (out.item(), ref)
