"""A wait inside a kernel that runs out (its bound set low through pssd_test_fault) ends the call with
PSSD_ERR_TIMEOUT instead of a wrong result; the handle then solves the problem normally."""
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


# k = 10 and 30: one leaf of one and of two block columns; 150: several leaves, tensor-core products
@pytest.mark.parametrize("k", [10, 30, 150])
@pytest.mark.parametrize("fault,precision", [("FAULT_LEAF64_WAIT", 0), ("FAULT_LEAF64_WAIT", 2), ("FAULT_LEAF32_WAIT", 1)])
def test_leaf_wait(P, k, fault, precision):
    H = torch.from_numpy(G.casida(k, ("uniform", 1.0, 10.0), seed=k)[0]).cuda()
    h = P.Handle()
    S, _ = P.sign(H, handle=h, precision=precision)
    h.test_fault(getattr(P, fault), 1)
    with pytest.raises(P.PssdError) as e:
        P.sign(H, handle=h, precision=precision)
    assert e.value.status == 5
    h.test_fault(getattr(P, fault), 0)
    S1, _ = P.sign(H, handle=h, precision=precision)
    assert torch.equal(S1, S)
    h.close()


@pytest.mark.parametrize("op,power", [(0, 0), (1, 0), (0, 20), (1, 20)])
def test_krylov_wait(P, op, power):
    """128 CTAs meet at a barrier for every product: with one poll each, CTA 0 gives up at one of them."""
    m = 1024
    g = torch.Generator(device="cuda"); g.manual_seed(m)
    A = torch.randn(m, m, device="cuda", dtype=torch.float64, generator=g)
    A = A @ A.T / m
    h = P.Handle()
    out, _ = P.test_krylov(A, op=op, power=power, seed=7, handle=h)
    h.test_fault(P.FAULT_KRYLOV_WAIT, 1)
    with pytest.raises(P.PssdError) as e:
        P.test_krylov(A, op=op, power=power, seed=7, handle=h)
    assert e.value.status == 5
    h.test_fault(P.FAULT_KRYLOV_WAIT, 0)
    again, _ = P.test_krylov(A, op=op, power=power, seed=7, handle=h)
    assert torch.equal(again, out)
    h.close()


@pytest.mark.parametrize("call", ["sign", "eig"])
def test_krylov_wait_in_a_call(P, call):
    H = torch.from_numpy(G.casida(300, ("uniform", 1.0, 10.0), seed=5)[0]).cuda()
    h = P.Handle()
    ref = getattr(P, call)(H, handle=h)
    h.test_fault(P.FAULT_KRYLOV_WAIT, 1)
    with pytest.raises(P.PssdError) as e:
        getattr(P, call)(H, handle=h)
    assert e.value.status == 5
    h.test_fault(P.FAULT_KRYLOV_WAIT, 0)
    assert torch.equal(getattr(P, call)(H, handle=h)[0], ref[0])
    h.close()
