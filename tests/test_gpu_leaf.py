"""The Cholesky leaves at the edges of their blocks (32 columns; 64 in FP64, 128 in FP32) through the sign of small
definite matrices, against the spectral definition."""
import numpy as np
import pytest
import torch

import casida_inputs as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2203_08900_gb300 import build as b
    b.build()
    import paper_2203_08900_gb300 as P
    P.lib()
    return P


def _sign(H, sigma):
    s = sigma.astype(float)
    L = np.linalg.cholesky(s[:, None] * H)
    w, Z = np.linalg.eigh(L.T @ (s[:, None] * L))
    return np.linalg.solve(L.T, (Z * np.sign(w)) @ Z.T @ L.T)


@pytest.mark.parametrize("n", [1, 2, 3, 16, 31, 32, 33, 47, 63, 64, 65, 96, 97, 127, 128, 129, 160, 191])
@pytest.mark.parametrize("precision", [0, 1, 2])
def test_sign_small(P, n, precision):
    H, sigma = G.example1(n, 10.0, seed=n)
    S, info = P.sign(torch.from_numpy(H).cuda(), sigma=sigma, precision=precision)
    ref = _sign(H, sigma)
    # FP64: a few hundred roundings amplified by the condition number 10 of Sigma H and by ||S||;
    # mixed: the FP32 iteration's error with the same factors
    tol = (1e-13 if precision != 1 else 1e-4) * max(1.0, np.linalg.norm(ref, 2)) ** 2
    assert np.linalg.norm(S.cpu().numpy() - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("bad", [0, 5, 31, 32, 40, 63, 64, 100])
def test_failing_pivot(P, bad):
    """The first pivot that is not positive is the one reported."""
    n = 110
    d = np.ones(n)
    d[bad:] = -1.0
    with pytest.raises(P.PssdError) as e:
        P.sign(torch.diag(torch.from_numpy(d)).cuda(), sigma=np.ones(n, dtype=np.int8))
    assert e.value.status == 1
