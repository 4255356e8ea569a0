"""The FP32 tensor-core product where its tile width changes: products of one and of several
rounds of tiles, wide ones, and triangular and lower-only ones whose operands are prepared for
their own triangle alone (what lies beyond it is set to NaN).  Bound: 3xTF32 drops A_lo B_lo and
rounds the parts, at most 2^-19 of |A||B| in all; FP32 accumulation of k terms adds k 2^-23."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2203_08900_gb300 import build as b
    b.build()
    import paper_2203_08900_gb300 as P
    P.lib()
    return P


# m, n, k, triA, triB, lowerC, batch: widths of 64 (304 tiles at most), 128 and 256
CASES = [
    (1200, 1900, 40, 0, 0, 0, 1),      # 300 tiles of 64
    (1281, 1900, 40, 0, 0, 0, 1),      # 330: wider ones
    (1000, 1030, 100, 0, 0, 1, 4),
    (769, 769, 769, 0, 2, 0, 4),
    (769, 769, 769, 2, 1, 1, 7),
    (2000, 2047, 24, 0, 0, 0, 2),      # 256 of 256
    (3073, 3100, 17, 0, 0, 1, 2),
]


@pytest.mark.parametrize("m,n,k,triA,triB,lowerC,batch", CASES)
def test_tile_widths(P, m, n, k, triA, triB, lowerC, batch):
    g = torch.Generator(device="cuda"); g.manual_seed(m + n + k)
    A = torch.randn(batch, m, k, device="cuda", generator=g)
    B = torch.randn(batch, k, n, device="cuda", generator=g)
    Cin = torch.randn(batch, m, n, device="cuda", generator=g)
    cut = {0: lambda X: X, 1: torch.tril, 2: torch.triu}
    A64, B64 = cut[triA](A).double(), cut[triB](B).double()
    for X, tri in ((A, triA), (B, triB)):
        if tri:
            outside = ~cut[tri](torch.ones_like(X, dtype=torch.bool))
            X[outside] = float("nan")
    alpha, beta = -0.75, 0.5
    C = P.test_gemm_f32(A, B, triA=triA, triB=triB, lowerC=lowerC, alpha=alpha, beta=beta, Cin=Cin).double()
    ref = alpha * (A64 @ B64) + beta * Cin.double()
    bound = (2.0 ** -19 + k * 2.0 ** -23) * (abs(alpha) * (A64.abs() @ B64.abs())) + 2.0 ** -22 * (beta * Cin.double().abs())
    err = (C - ref).abs()
    if lowerC:
        err, bound = err.tril(), bound.tril()
    assert bool((err <= bound + 1e-30).all()), float((err / (bound + 1e-30)).max())
