"""The two halves of a division side by side when something fails on the host (pssd_test_fault): what the second
half's thread meets is reported as it would be on the calling thread, and the handle stays usable."""
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


def _H(k, seed=11):
    return torch.from_numpy(G.casida(k, ("uniform", 1.0, 10.0), seed=seed)[0]).cuda()


@pytest.mark.parametrize("call", ["eig", "casida_eig"])
def test_refused_launch_in_the_second_half_is_reported(P, call):
    H = _H(200)
    k = H.shape[0] // 2
    blocks = H[:k, :k].contiguous(), H[:k, k:].contiguous()
    h = P.Handle()
    run = lambda: P.eig(H, handle=h) if call == "eig" else P.casida_eig(*blocks, handle=h)   # noqa: E731
    D, V, _ = run()
    h.test_fault(P.FAULT_LAUNCH, 1)
    with pytest.raises(P.PssdError) as e:
        run()
    assert e.value.status == 6 and "kernel launch" in str(e.value)
    h.test_fault(P.FAULT_LAUNCH, 0)
    D1, V1, _ = run()
    assert torch.equal(D1, D) and torch.equal(V1, V)
    h.close()


@pytest.mark.parametrize("fault,value,launch", [("FAULT_MEMORY", 1 << 30, 1), ("FAULT_STREAM", 1, 2)])
def test_refused_launch_survives_a_refused_helper(P, fault, value, launch):
    """A second half without memory or stream runs in the first one's chain; a launch refused before is reported all
    the same."""
    H = _H(200)
    h = P.Handle()
    h.test_fault(getattr(P, fault), value)      # (1 GiB: the handle's own workspace, nothing for a helper)
    D, V, _ = P.eig(H, handle=h)
    h.test_fault(P.FAULT_LAUNCH, launch)
    with pytest.raises(P.PssdError) as e:
        P.eig(H, handle=h)
    assert e.value.status == 6
    h.test_fault(P.FAULT_LAUNCH, 0)
    D1, V1, _ = P.eig(H, handle=h)
    assert torch.equal(D1, D) and torch.equal(V1, V)
    h.close()


MIB = 1 << 20


def _program(P, cap, side_by_side, kind, H, h=None):
    """The outputs of a program whose last call may use `cap` bytes of workspace (0: no limit); None if they are too
    few.  Pieces of 1 MiB, so that what is held follows what is needed."""
    k = H.shape[0] // 2
    own = h is None
    if own:
        h = P.Handle()
        h.test_fault(P.FAULT_CHUNK, MIB)
        h.test_fault(P.FAULT_STREAM, 0 if side_by_side else 1)
    if kind == "eig then split":
        P.eig(H, handle=h)
    h.test_fault(P.FAULT_MEMORY, cap)
    try:
        if kind == "eig":
            out = P.eig(H, handle=h)[:2]
        elif kind == "casida_eig":
            out = P.casida_eig(H[:k, :k].contiguous(), H[:k, k:].contiguous(), handle=h)[:2]
        else:
            out = P.split(H, r=8, handle=h, precision=P.PSSD_FP64_EMULATED)[:3]
    except P.PssdError as e:
        assert e.status == 7
        out = None
    h.test_fault(P.FAULT_MEMORY, 0)
    if own:
        h.close()
    return out


@pytest.mark.parametrize("kind", ["eig", "casida_eig", "eig then split"])
def test_what_fits_in_sequence_fits_side_by_side(P, kind):
    """The least memory with which a program runs without helpers is enough with them, and so is anything between
    that and what it takes undisturbed; the results are the same to the bit."""
    H = _H(260)
    ref = _program(P, 0, False, kind, H)
    lo, hi = 0, 4096                                 # MiB: too little, enough
    assert _program(P, hi * MIB, False, kind, H) is not None
    while hi - lo > 1:
        mid = (lo + hi) // 2
        if _program(P, mid * MIB, False, kind, H) is None:
            lo = mid
        else:
            hi = mid
    for cap in [hi * MIB + d * MIB for d in (0, 1, 2, 3, 4, 6, 8, 12, 16, 24, 32, 64, 128)] + [0]:
        out = _program(P, cap, True, kind, H)
        assert out is not None, (hi, cap // MIB)
        assert all(torch.equal(x, y) for x, y in zip(out, ref)), cap // MIB


def test_helpers_keep_little_between_calls(P):
    """After a large call the helpers hold 1 GiB each at most beside what the handle keeps without them."""
    n = 8192
    g = torch.Generator(device="cuda"); g.manual_seed(2)
    B = torch.randn(n, n, device="cuda", dtype=torch.float64, generator=g)
    M = B @ B.T / n + torch.eye(n, device="cuda", dtype=torch.float64)
    s = torch.ones(n, device="cuda", dtype=torch.float64)
    s[1::2] = -1.0
    H, sigma = s[:, None] * (0.5 * (M + M.T)), s.cpu().numpy()
    del B, M
    small = _H(200)
    kept = []
    for refused in (1, 0):
        h = P.Handle()
        h.test_fault(P.FAULT_STREAM, refused)
        P.eig(small, handle=h)                       # (loads the kernels)
        P.eig(H, sigma=sigma, handle=h, precision=P.PSSD_FP64_EMULATED)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        before = torch.cuda.mem_get_info()[0]
        h.close()
        kept.append(torch.cuda.mem_get_info()[0] - before)
    assert kept[1] - kept[0] <= 3 * 1024 * MIB + 64 * MIB, kept


def test_profiled_calls_reuse_their_events(P):
    """The timing events of the second halves go back to the pools they came from: ten more calls make fewer events
    than the first one did."""
    H = _H(200)
    h = P.Handle()
    h.profile(True)
    n0 = P.timing_event_count()
    P.eig(H, handle=h)
    n1 = P.timing_event_count()
    for _ in range(10):
        P.eig(H, handle=h)
    assert P.timing_event_count() - n1 < n1 - n0
    h.close()
