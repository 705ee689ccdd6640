"""GPU parity of the FP64 whole-block groups where one grid is shared by a
cluster of blocks: each block owns a slab of the longest axis, so what can go
wrong sits at the slabs' edges, at the split axis (a rate, V), in axes shorter
than the cluster and in lines longer than a slab.

The bounds are those of the other FP64 paths (1e-12 of the largest value of a
grid, node by node: some 1e3 roundings of 1e-16 in a row of a line solve).
"""
import numpy as np
import pytest

from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from paper_2408_00559_gb300 import workloads as W
from test_gpu_parity import TOL64, check_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


CASES = [
    # (N, level, full, payoff, boundary condition)
    (2, 4, True, "caplet", "neumann"),      # 256 nodes: two blocks
    (2, 5, True, "caplet", "neumann"),      # 1024 nodes: eight blocks of 4 rows
    (2, 5, True, "caplet", "dirichlet"),
    (2, 8, False, "caplet", "neumann"),     # split along the rate, then along V
    (2, 8, False, "caplet", "dirichlet"),
    (2, 10, False, "caplet", "neumann"),    # lines of 1024 rows
    (3, 4, True, "swaption", "neumann"),    # 4096 nodes
    (3, 4, True, "swaption", "dirichlet"),
    (5, 2, True, "swaption", "neumann"),    # axes of 4 rows: four blocks at most
    (8, 1, True, "swaption", "neumann"),    # axes of 2 rows: two blocks
]


@pytest.mark.parametrize("case", CASES, ids=[f"N{c[0]}_n{c[1]}{'_full' if c[2] else ''}_{c[4]}" for c in CASES])
def test_clusters_match_oracle(case):
    N, n, full, payoff, bc = case
    inst = W.small_instance(N, n, steps=3, seed=900 + N * 10 + n, full=full, payoff=payoff)
    check_problem(dict(inst, bc=bc), TOL64, TOL64)


def test_one_block_per_grid_equals_clusters():
    # 200 grids leave no blocks to spare: the same grids without clusters
    insts = [dict(W.small_instance(2, 5, steps=3, seed=s, full=True, payoff="caplet")) for s in range(200)]
    p = B.solve_batch(insts)
    for i in (0, 77, 199):
        prob = B.Problem(insts[i])
        prob.step(1)
        prob.step(2)
        one = prob.combine()
        assert abs(one - p[i]) <= TOL64 * abs(p[i]), (i, one, p[i])
        prob.close()
