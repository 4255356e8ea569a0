"""The slice engine's operand preparation (test hook engine 2) at the edges of its bands of 16 rows and k blocks of
16, for every operand structure, odd leading dimensions and all-zero, subnormal and huge rows."""
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


@pytest.mark.parametrize("m,n,k,batch", [(1, 1, 1, 1), (15, 17, 16, 2), (130, 66, 15, 1), (129, 129, 129, 3),
                                         (300, 300, 300, 1), (64, 700, 513, 1)])
@pytest.mark.parametrize("ta,tb,triA,triB,lowerC,ks", [
    (0, 0, 0, 0, 0, False), (1, 0, 0, 0, 1, False), (0, 1, 0, 0, 0, True), (1, 1, 0, 0, 1, False),
    (0, 1, 0, 2, 0, False), (0, 0, 1, 0, 0, False), (1, 0, 2, 1, 1, True), (1, 1, 1, 2, 0, False)])
def test_prepared_operands(P, m, n, k, batch, ta, tb, triA, triB, lowerC, ks):
    g = torch.Generator(device="cuda"); g.manual_seed(m + 3 * n + 7 * k)
    r = lambda *s: torch.randn(*s, device="cuda", dtype=torch.float64, generator=g)   # noqa: E731
    rows = torch.ones(m, device="cuda", dtype=torch.float64)
    for i, f in enumerate((0.0, 1e-310, 1e250)):          # one row of each kind
        if m > 3:
            rows[(i * 7 + 2) % m] = f
    A = r(batch, m, k) * rows[None, :, None]
    A = A.mT.contiguous() if ta else A
    B = r(batch, n if tb else k, k if tb else n)
    scale = (torch.randint(0, 2, (k,), device="cuda", generator=g).double() * 2 - 1) if ks else None
    C = P.test_gemm_f64(A, B, engine=2, ta=ta, tb=tb, triA=triA, triB=triB, lowerC=lowerC, kscale=scale)
    tri = {0: lambda X: X, 1: torch.tril, 2: torch.triu}
    opA, opB = tri[triA](A.mT if ta else A), tri[triB](B.mT if tb else B)
    ref = (opA * scale if ks else opA) @ opB
    # 56 bits of each row's and column's largest entry, sums in 48-bit pairs; a subnormal row has
    # the accuracy of its last bit
    bound = 2.0 ** -46 * k * opA.abs().amax(-1, keepdim=True) * opB.abs().amax(-2, keepdim=True) + 1e-321 * k
    err = (C - ref).abs() - bound
    assert float((torch.tril(err) if lowerC else err).max()) <= 0.0
