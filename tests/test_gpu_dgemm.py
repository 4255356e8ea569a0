"""The FP64-pipe GEMM (test hook engine 0) at the edges of its tiles -- orders 8, 16 and 32, k blocks of 64, 32
and 16 -- for every operand structure, against torch's FP64 product."""
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


SIZES = [
    # m, n, k, batch: 8 x 8 tiles (k split four ways), 16 x 16 and 32 x 32
    (1, 1, 1, 1), (7, 9, 3, 2), (8, 8, 64, 1), (17, 15, 65, 3), (33, 100, 129, 1), (100, 33, 31, 1),
    (250, 250, 33, 1), (255, 257, 32, 2), (700, 690, 17, 3), (1217, 1217, 40, 1),
]
FORMS = [
    # ta, tb, triA, triB, lowerC, kscale, beta
    (0, 0, 0, 0, 0, False, 0.0), (1, 0, 0, 0, 1, False, 0.0), (0, 1, 0, 0, 1, True, -1.0), (1, 1, 0, 0, 0, False, 0.5),
    (0, 1, 0, 2, 0, False, 0.0), (0, 0, 1, 0, 0, False, 1.0), (1, 0, 2, 1, 1, True, 0.0), (0, 0, 2, 2, 0, False, 0.0),
]


@pytest.mark.parametrize("m,n,k,batch", SIZES)
@pytest.mark.parametrize("ta,tb,triA,triB,lowerC,ks,beta", FORMS)
def test_dgemm(P, m, n, k, batch, ta, tb, triA, triB, lowerC, ks, beta):
    g = torch.Generator(device="cuda"); g.manual_seed(m * 7 + n * 3 + k)
    r = lambda *s: torch.randn(*s, device="cuda", dtype=torch.float64, generator=g)   # noqa: E731
    A = r(batch, k if ta else m, m if ta else k)
    B = r(batch, n if tb else k, k if tb else n)
    Cin = r(batch, m, n)
    scale = (torch.randint(0, 2, (k,), device="cuda", generator=g).double() * 2 - 1) if ks else None
    C = P.test_gemm_f64(A, B, engine=0, ta=ta, tb=tb, triA=triA, triB=triB, lowerC=lowerC, alpha=0.75, beta=beta,
                        Cin=Cin, kscale=scale)
    tri = {0: lambda X: X, 1: torch.tril, 2: torch.triu}
    opA, opB = tri[triA](A.mT if ta else A), tri[triB](B.mT if tb else B)
    ref = 0.75 * ((opA * scale if ks else opA) @ opB) + beta * Cin
    # k roundings of each side's sum and a few of the scaling, u = 2^-53
    bound = 2.0 ** -53 * ((2 * k + 8) * (opA.abs() @ opB.abs()) + 8 * abs(beta) * Cin.abs())
    err = (C - ref).abs() - bound
    assert float((torch.tril(err) if lowerC else err).max()) <= 0.0
