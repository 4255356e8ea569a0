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
