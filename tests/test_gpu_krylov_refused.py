"""Krylov loops whose cooperative launch is refused (as on a part of the GPU too small for all of its CTAs; made
with pssd_test_fault) run step by step instead."""
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


@pytest.mark.parametrize("op,power", [(0, 0), (1, 0), (0, 20), (1, 20)])
@pytest.mark.parametrize("m", [30, 1024])
def test_refused_loop_runs_step_by_step(P, m, op, power):
    g = torch.Generator(device="cuda"); g.manual_seed(m)
    A = torch.randn(m, m, device="cuda", dtype=torch.float64, generator=g)
    A = A @ A.T / m
    kw = dict(op=op, power=power, seed=7)
    ref, _ = P.test_krylov(A, fused=False, **kw)
    h = P.Handle()
    h.test_fault(P.FAULT_KRYLOV_LAUNCH, 1)
    out, _ = P.test_krylov(A, fused=True, handle=h, **kw)
    assert torch.equal(out, ref)
    h.close()


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_calls_without_the_fused_loops(P, precision):
    """The loops only estimate bounds and shifts: the results are those of the fused loops to the mode's accuracy."""
    H = torch.from_numpy(G.casida(150, ("uniform", 1.0, 10.0), seed=5)[0]).cuda()
    h = P.Handle()
    S, _ = P.sign(H, handle=h, precision=precision)
    D, _, _ = P.eig(H, handle=h, precision=precision)
    h.test_fault(P.FAULT_KRYLOV_LAUNCH, 1)
    S1, _ = P.sign(H, handle=h, precision=precision)
    D1, _, _ = P.eig(H, handle=h, precision=precision)
    # condition numbers below 10 each for the sign and the congruence, FP64 or the FP32 iteration
    tol = 1e-11 if precision != 1 else 1e-3
    assert float(torch.linalg.norm(S1 - S) / torch.linalg.norm(S)) <= tol
    assert float((D1 - D).abs().max() / D.abs().max()) <= tol
    h.close()
