"""The Jacobi leaf (orders up to 64, through the symmetric recursion's test hook without refinement): residual and
orthogonality on random, graded, clustered, diagonal, zero and far-scaled matrices."""
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


def _matrix(kind, m, g):
    r = lambda *s: torch.randn(*s, device="cuda", dtype=torch.float64, generator=g)   # noqa: E731
    Q = torch.linalg.qr(r(m, m))[0]
    if kind == "random":
        d = r(m)
    elif kind == "graded":
        d = torch.logspace(-14, 2, m, device="cuda", dtype=torch.float64)
    elif kind == "clustered":
        d = 1.0 + 1e-9 * r(m)
    elif kind == "diagonal":
        return torch.diag(r(m))
    elif kind == "zero":
        return torch.zeros(m, m, device="cuda", dtype=torch.float64)
    else:
        d = 1e-200 * r(m)
    B = (Q * d) @ Q.T
    return 0.5 * (B + B.T)


@pytest.mark.parametrize("m", [1, 2, 3, 16, 31, 48, 63, 64])
@pytest.mark.parametrize("kind", ["random", "graded", "clustered", "diagonal", "zero", "small"])
def test_jacobi_leaf(P, m, kind):
    g = torch.Generator(device="cuda"); g.manual_seed(m)
    B = _matrix(kind, m, g)
    w, W, _ = P.test_sym_eig(B, flags=P.FLAG_NO_REFINE)
    s = max(float(B.abs().max()), 1e-300)
    # a column takes part in fewer than 4 * 63 FP64 rotations of three roundings each, 2^-53
    tol = 4 * 63 * 3 * 2.0 ** -53
    assert float(torch.linalg.norm(W.T @ W - torch.eye(m, device="cuda", dtype=torch.float64))) <= tol * m ** 0.5
    assert float(torch.linalg.norm(B / s @ W - W * (w / s))) <= tol * max(1.0, float(torch.linalg.norm(B / s)))
