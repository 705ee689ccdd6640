"""Batches in which some grids are solved as bundles and some by the warp groups:
every instance is priced as it is alone, and the launches are counted, so that
bundles do run (a batch with both has one launch more than one without).

What is left to the warp groups: three instances beyond the last full bundle,
and instances with Dirichlet faces, alternating with the others or most of the
book.  Counts follow the rule (4000 Inner nodes per SM in mixed precision, 1300
in FP64).  Prices: a component value may move by a few ulps of FP64 (64 of them
allowed), the price by kappa = sum |c_l u_l| / |price| times that.
"""
import numpy as np
import pytest

from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from paper_2408_00559_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NODES_PER_SM = {"mixed": 4000, "fp64": 1300}


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


def instances(N, level, count, precision, bc):
    out = [W.small_instance(N, level, steps=2, seed=7000 + s, precision=precision,
                            payoff="caplet" if N == 2 else "swaption") for s in range(count)]
    return [dict(x, bc=bc(k)) for k, x in enumerate(out)]


def neumann(k):
    return "neumann"


def enough(N, level, precision):
    """Instances of one shape, a multiple of 32, that make bundles worth while."""
    import torch
    prob = B.Problem(W.small_instance(N, level, steps=1, precision=precision))
    sizes = 2 ** prob.grid_info()[0].sum(axis=1)
    prob.close()
    need = NODES_PER_SM[precision] * torch.cuda.get_device_properties(0).multi_processor_count
    return -(-need // int(sizes[sizes <= 64].sum())) // 32 * 32 + 32


def run(insts):
    import torch
    b = B.Batch(insts)
    b.set_kappa_max(0)
    out = torch.zeros(len(insts), dtype=torch.float64, device="cuda")
    b.run(out.data_ptr())
    torch.cuda.synchronize()
    n = b.launches()
    b.close()
    return out.cpu().numpy(), n


def alone(inst):
    """Price and kappa of one instance on the warp groups."""
    prob = B.Problem(inst)
    prob.step(inst["n_steps"])
    p = prob.combine()
    scale = np.sum(np.abs(prob.grid_info()[1] * prob.grid_values())) * inst.get("discount", 1.0)
    prob.close()
    return p, scale / abs(p)


def check(insts, prices, picks):
    assert np.all(np.isfinite(prices))
    for k in picks:
        p, kappa = alone(insts[k])
        assert abs(prices[k] - p) <= 64 * 2.2e-16 * max(kappa, 1.0) * abs(p), (k, prices[k], p, kappa)


def test_few_bundles_in_a_dirichlet_book():
    book = instances(4, 5, 417, "fp64", lambda k: "dirichlet" if k < 400 else "neumann")
    prices, n = run(book)
    assert n == 3, n  # bundles of 17, the warp groups, the combination
    check(book, prices, (0, 399, 400, 416))


@pytest.mark.parametrize("N,level,precision", [(2, 6, "mixed"), (3, 6, "mixed"), (3, 6, "fp64"), (4, 6, "fp64"),
                                               (8, 4, "mixed")])
def test_bundles_with_leftovers(N, level, precision):
    count = enough(N, level, precision) + 3
    insts = instances(N, level, count, precision, neumann)
    prices, n = run(insts)
    assert n == 3, n  # bundles, the three left over, the combination
    check(insts, prices, (0, 31, count // 2, count - 4, count - 1))


@pytest.mark.parametrize("N,level,precision", [(3, 5, "mixed"), (4, 5, "fp64")])
def test_bundles_beside_dirichlet_instances(N, level, precision):
    count = 2 * enough(N, level, precision)
    insts = instances(N, level, count, precision, lambda k: "dirichlet" if k % 2 else "neumann")
    prices, n = run(insts)
    assert n == 3, n
    check(insts, prices, (0, 1, count // 2, count // 2 + 1, count - 2, count - 1))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_noalloc_up_to_its_array_with_and_without_bundles(precision):
    # the fixed array holds the records, the grid list and, if they still fit,
    # the lists of bundles; at the limit the call plans again without those
    import torch
    one = instances(4, 5, 1, precision, neumann)
    b = B.Batch(one)
    grids = 121
    record = b.io_bytes()[0] - 40 * grids
    b.close()
    room = 16 << 20

    def used(n):
        up = lambda x: -(-x // 256) * 256  # noqa: E731
        return up(record * n) + up(32 * grids * n) + 2 * up(8 * grids * n) + 3 * 256

    most = room // (record + 48 * grids)
    while used(most) > room:
        most -= 1
    insts = instances(4, 5, most + 2, precision, neumann)
    out = torch.zeros(most + 2, dtype=torch.float64, device="cuda")
    for n in (most // 2, most):
        out.fill_(float("nan"))
        B.solve_noalloc(insts[:n], out.data_ptr())
        torch.cuda.synchronize()
        check(insts, out[:n].cpu().numpy(), (0, 33, n - 1))
    with pytest.raises(B.AmfrwError) as e:
        B.solve_noalloc(insts, out.data_ptr())
    assert e.value.status == 7
