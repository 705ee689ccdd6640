"""Bundles: grids of one shape from many instances, one instance per lane.

A batch large enough for bundles must price every instance like the warp
groups that price it in a small batch.  In mixed precision both run the same
FP32 operations in the same order, so only the FP64 interpolation and sums
differ; in FP64 the stencil and the line solves are associated differently.
Either way a component value moves by a few ulps of FP64, so a price by that
times its cancellation kappa = sum |c_l u_l| / |sum c_l u_l| (the instance's
own in mixed precision, where the batch reports it; 1e4 in FP64).  The shapes cover every node block
(axes of 2, 4, 8 and more rows, on rates and on V), grids of 1 to 64 nodes,
full and partial bundles and the left-over instances.
"""
import numpy as np
import pytest

from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD
from paper_2408_00559_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


def prices(insts):
    import torch
    b = B.Batch(insts)
    b.set_kappa_max(1e300 if insts[0]["precision"] == "mixed" else 0)
    out = torch.zeros(len(insts), dtype=torch.float64, device="cuda")
    b.run(out.data_ptr())
    torch.cuda.synchronize()
    kappa = b.promoted()[1]
    launches = b.launches()
    b.close()
    return out.cpu().numpy(), kappa, launches


@pytest.mark.parametrize("N,level,count,full,payoff,precision", [
    (2, 6, 1100, False, "caplet", "mixed"), (2, 6, 500, False, "caplet", "fp64"),
    (3, 6, 205, False, "swaption", "mixed"), (3, 6, 82, False, "swaption", "fp64"),
    (4, 6, 78, False, "swaption", "mixed"), (4, 6, 52, False, "caplet", "fp64"),
    (8, 4, 109, False, "swaption", "mixed"), (8, 4, 50, False, "swaption", "fp64"),
    (6, 1, 9600, True, "swaption", "mixed"), (2, 3, 3200, True, "swaption", "fp64"),
])
def test_bundles_price_like_warp_groups(N, level, count, full, payoff, precision):
    insts = [W.small_instance(N, level, steps=2, seed=s, precision=precision, full=full, payoff=payoff)
             for s in range(count)]
    got, kappa, n_big = prices(insts)
    pick = list(range(0, count, max(1, count // 9)))[:9] + [count - 1]
    ref, kref, _ = prices([insts[i] for i in pick])
    scale = np.maximum(kref if precision == "mixed" else 1e4, 1.0)
    err = np.abs(got[pick] - ref) / np.abs(ref)
    assert np.all(np.isfinite(got))
    assert np.all(err <= 64 * 2.2e-16 * scale), (err.max(), scale[err.argmax()] if np.ndim(scale) else scale)
