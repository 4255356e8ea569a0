"""The float-pair product on tiles of 16, taken by small products with k <= 128, holds the bits of the one on tiles
of 64, which the same product takes in a batch of 39 copies."""
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


@pytest.mark.parametrize("m,n,k,ta,tb,triA,triB,lowerC", [
    (1, 1, 1, 0, 0, 0, 0, 0),
    (16, 17, 15, 0, 0, 0, 0, 0),
    (33, 64, 128, 1, 0, 0, 0, 0),
    (64, 31, 129, 0, 1, 0, 0, 0),      # beyond the rule: tiles of 64 on both sides
    (47, 47, 47, 0, 0, 1, 2, 0),
    (64, 63, 63, 0, 1, 0, 2, 0),
    (63, 63, 63, 1, 0, 2, 1, 1),
    (64, 64, 100, 0, 1, 0, 0, 1),
])
def test_tiles_agree(P, m, n, k, ta, tb, triA, triB, lowerC):
    g = torch.Generator(device="cuda"); g.manual_seed(m + 64 * n + k)
    A = torch.randn(k if ta else m, m if ta else k, device="cuda", dtype=torch.float64, generator=g)
    B = torch.randn(n if tb else k, k if tb else n, device="cuda", dtype=torch.float64, generator=g)
    copies = lambda X: X.expand(39, *X.shape).contiguous()
    kw = dict(engine=1, ta=ta, tb=tb, triA=triA, triB=triB, lowerC=lowerC, alpha=-0.75)
    one = P.test_gemm_f64(A, B, **kw)
    many = P.test_gemm_f64(copies(A), copies(B), **kw)
    if lowerC:
        one, many = one.tril(), many.tril()
    assert torch.equal(many, copies(one))
