"""The tensor-core GEMM at the edges of its tiles: one chunk of K (whose stage
is smaller than the epilogue's buffers, which reach past it), a remainder of a
chunk, more chunks than stages, every kind of tile width and ragged rows.

BF16 products are exact in FP32; K of them are added, each addition off by at
most 2^-23 of the sum of magnitudes (one unit in the last place, rounded either
way): the bound below, element by element, against FP64.
"""
import pytest

from paper_2408_00559_gb300 import _lib as B
from paper_2408_00559_gb300 import build as BLD

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    BLD.build()
    B.lib()


@pytest.mark.parametrize("K", [16, 64, 80, 720])
@pytest.mark.parametrize("M,N", [(1, 16), (1000, 48), (333, 80), (10245, 128), (129, 144), (10245, 160), (700, 512)])
def test_tile_edges(M, N, K):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + 31 * N + 7 * K)
    A = torch.randn(M, K, device="cuda", generator=g).to(torch.bfloat16)
    Bm = torch.randn(N, K, device="cuda", generator=g).to(torch.bfloat16)
    C = torch.full((M, N), float("nan"), device="cuda", dtype=torch.float32)
    for _ in range(3):
        B.tc_gemm_bf16(A, Bm, C)
        ref = A.double() @ Bm.double().T
        bound = K * 2.0 ** -23 * (A.double().abs() @ Bm.double().abs().T)
        assert bool(((C.double() - ref).abs() <= bound).all()), (C.double() - ref).abs().max().item()
        C.fill_(float("nan"))
