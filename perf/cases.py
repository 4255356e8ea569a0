"""The work that users of this framework have it do, as cases for timing and for comparing outputs.

Each case is one call (or one batch) through the public entry points of
``paper_2203_08900_gb300`` on seeded synthetic matrices: the Casida form
(A = (P + R)/2, B = (P - R)/2 with prescribed spectra of P and R), the
Example-1 form (random signature, spectrum equally spaced in [1, kappa]), the
complex BSE2 form and general pseudosymmetric matrices with a built-in
spectrum.  The random orthogonal factors are products of two orthonormal
Hartley transforms with random diagonal signs in between (dense, any order,
made with FFTs in a fraction of a second where a QR would take seconds).
"""
import math

import numpy as np
import torch

import paper_2203_08900_gb300 as P

PRECISION = {"fp64": P.PSSD_FP64, "fp64e": P.PSSD_FP64_EMULATED, "mixed": P.PSSD_MIXED}


def listed():
    return [
        # the smallest call of a program that knows its bounds' scale: the order-128 sign of the accuracy tests
        {"name": "sign_n128_fp64", "kind": "sign", "n": 128, "precision": "fp64", "r": 8, "dist": "u1_10"},
        # the allocation-free entry point inside a loop that owns its memory; not a multiple of any tile
        {"name": "noalloc_n90_fp64e", "kind": "noalloc", "n": 90, "precision": "fp64e", "r": 0, "dist": "u1_10"},
        # a whole small diagonalisation of the paper's Example 1: odd order, random signature, native FP64
        {"name": "eig_n251_fp64", "kind": "eig", "n": 251, "precision": "fp64", "kappa": 100.0},
        # the fast sign of a mid-sized matrix inside a larger program, ragged order
        {"name": "sign_n1000_mixed", "kind": "sign", "n": 1000, "precision": "mixed", "r": 0, "dist": "u0.1_100"},
        # the ordinary spectral division: one split of an order-4096 Casida matrix
        {"name": "split_n4096_mixed", "kind": "split", "n": 4096, "precision": "mixed", "dist": "u0.1_100"},
        # the benchmark's split (its distribution and precision) at the largest order that fits a short pass
        {"name": "split_n12288_mixed", "kind": "split", "n": 12288, "precision": "mixed", "dist": "log1e-2_1e2"},
        # the FP64-accurate split, the mode that meets the method's FP64 targets
        {"name": "split_n8192_fp64e", "kind": "split", "n": 8192, "precision": "fp64e", "dist": "log1e-2_1e2"},
        # a gradient through the sign (forward and step reversal) as in training on <G, S> + sum of positive eigenvalues
        {"name": "vjp_n2048_fp64", "kind": "vjp", "n": 2048, "precision": "fp64", "dist": "u1_10"},
        # the structure-aware split of a large Casida problem given by its blocks, ragged order
        {"name": "casida_split_k3000_fp64e", "kind": "casida_split", "k": 3000, "precision": "fp64e",
         "dist": "log1e-2_1e2"},
        # the structure-aware full diagonalisation (excitation energies and vectors)
        {"name": "casida_eig_k1024_fp64e", "kind": "casida_eig", "k": 1024, "precision": "fp64e", "dist": "u0.5_50"},
        # many Hamiltonians of uneven sizes in one call, as in a scan over geometries
        {"name": "batch20_mixed", "kind": "batch", "count": 20, "k_lo": 16, "k_hi": 512, "precision": "mixed",
         "dist": "u0.5_50"},
        # a complex Bethe-Salpeter matrix, full diagonalisation
        {"name": "zeig_n400_fp64e", "kind": "zeig", "n": 400, "precision": "fp64e", "dist": "u1_10"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds: sizes log-uniform over each kind's range, odd and ragged ones included, and
    spectra over one to four decades."""
    kind = rng.choice(["sign", "noalloc", "eig", "split", "vjp", "casida_split", "casida_eig", "batch", "zeig"])
    lo = rng.choice([0.1, 0.5, 1.0])
    near = "u%g_%g" % (lo, lo * _log_int(rng, 10, 100))
    far = "log%g_%g" % (0.01 * _log_int(rng, 1, 10), 10 * _log_int(rng, 1, 10))
    if kind == "sign":
        prec = rng.choice(["fp64", "fp64e", "mixed"])
        return {"kind": kind, "n": 2 * _log_int(rng, 32, 512 if prec == "fp64" else 1536), "precision": prec,
                "r": rng.choice([0, 8]) if prec != "mixed" else 0, "dist": near}
    if kind == "noalloc":
        return {"kind": kind, "n": 2 * _log_int(rng, 8, 64), "precision": rng.choice(["fp64", "fp64e", "mixed"]), "r": 0,
                "dist": near}
    if kind == "eig":
        return {"kind": kind, "n": _log_int(rng, 65, 800), "precision": rng.choice(["fp64", "fp64e"]),
                "kappa": float(_log_int(rng, 10, 100))}
    if kind == "split":
        return {"kind": kind, "n": 2 * _log_int(rng, 256, 2800), "precision": rng.choice(["fp64e", "mixed"]),
                "dist": rng.choice([near, far])}
    if kind == "vjp":
        return {"kind": kind, "n": 2 * _log_int(rng, 64, 600), "precision": rng.choice(["fp64", "fp64e"]), "dist": near}
    if kind == "casida_split":
        return {"kind": kind, "k": _log_int(rng, 100, 3000), "precision": "fp64e", "dist": rng.choice([near, far])}
    if kind == "casida_eig":
        return {"kind": kind, "k": _log_int(rng, 100, 700), "precision": "fp64e", "dist": near}
    if kind == "batch":
        return {"kind": kind, "count": rng.randrange(4, 25), "k_lo": 16, "k_hi": _log_int(rng, 48, 400),
                "precision": rng.choice(["fp64e", "mixed"]), "dist": near}
    return {"kind": "zeig", "n": 2 * _log_int(rng, 40, 240), "precision": "fp64e", "dist": near}


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _spectrum(g, k, dist):
    u = torch.rand(k, generator=g, device="cuda", dtype=torch.float64)
    if dist.startswith("log"):
        lo, hi = (math.log(float(x)) for x in dist[3:].split("_"))
        return torch.exp(lo + (hi - lo) * u)
    lo, hi = (float(x) for x in dist[1:].split("_"))
    return lo + (hi - lo) * u


def _signs(g, k):
    return torch.randint(0, 2, (k,), generator=g, device="cuda", dtype=torch.int64).double() * 2 - 1


def _hartley(X):
    F = torch.fft.fft(X, dim=0)
    return (F.real - F.imag) / math.sqrt(X.shape[0])


def _symmetric(g, d):
    """Q diag(d) Q^T with Q = D1 F D2 F (F the orthonormal Hartley transform, D random signs)."""
    k = d.numel()
    s1, s2 = _signs(g, k), _signs(g, k)

    def q(X):
        return s1[:, None] * _hartley(s2[:, None] * _hartley(X))

    M = q(q(torch.diag(d)).T.contiguous())
    return (0.5 * (M + M.T)).contiguous()


def _blocks(g, k, dist):
    """A, B of the Casida form with spectra drawn from dist for A + B and A - B."""
    Pm, R = _symmetric(g, _spectrum(g, k, dist)), _symmetric(g, _spectrum(g, k, dist))
    return (0.5 * (Pm + R)).contiguous(), (0.5 * (Pm - R)).contiguous()


def _casida(g, k, dist):
    A, B = _blocks(g, k, dist)
    H = torch.empty(2 * k, 2 * k, device="cuda", dtype=torch.float64)
    H[:k, :k] = A
    H[:k, k:] = B
    H[k:, :k] = -B
    H[k:, k:] = -A
    return H


def _example1(g, n, kappa):
    sigma = _signs(g, n)
    M = _symmetric(g, torch.linspace(1.0, kappa, n, device="cuda", dtype=torch.float64))
    return (sigma[:, None] * M).contiguous(), sigma.cpu().numpy().astype(np.int8)


def _hermitian(g, d):
    """Q diag(d) Q^H with Q = D1 F D2 F (F the unitary Fourier transform, D random phases)."""
    k = d.numel()
    t1, t2 = (torch.exp(2j * math.pi * torch.rand(k, generator=g, device="cuda", dtype=torch.float64)) for _ in range(2))

    def q(X):
        return t1[:, None] * torch.fft.fft(t2[:, None] * torch.fft.fft(X, dim=0, norm="ortho"), dim=0, norm="ortho")

    M = q(q(torch.diag(d.to(torch.complex128))).mH.contiguous())
    return 0.5 * (M + M.mH)


def _bse2(g, n, dist):
    k = n // 2
    Pm, R = _hermitian(g, _spectrum(g, k, dist)), _hermitian(g, _spectrum(g, k, dist))
    A, B = 0.5 * (Pm + R), 0.5 * (Pm - R)
    return torch.cat([torch.cat([A, B], 1), torch.cat([-B, -A], 1)], 0).contiguous()


def _batch_orders(case):
    r = np.random.default_rng(case["count"])   # the sizes belong to the case, the matrices to the seed
    lo, hi = math.log(case["k_lo"]), math.log(case["k_hi"])
    return [int(round(math.exp(x))) for x in r.uniform(lo, hi, case["count"])]


def prepare(case, seed):
    g = _generator(seed)
    s = {"case": case, "kw": {"precision": PRECISION[case["precision"]]}}
    if case.get("r"):
        s["kw"]["r"] = case["r"]
    kind = case["kind"]
    if kind in ("sign", "noalloc", "split", "vjp"):
        s["H"] = _casida(g, case["n"] // 2, case["dist"])
        if kind == "noalloc":
            s["S"] = torch.empty_like(s["H"])
        if kind == "vjp":
            s["G"] = torch.randn(case["n"], case["n"], generator=g, device="cuda", dtype=torch.float64)
    elif kind == "eig":
        s["H"], s["sigma"] = _example1(g, case["n"], case["kappa"])
    elif kind in ("casida_split", "casida_eig"):
        s["A"], s["B"] = _blocks(g, case["k"], case["dist"])
    elif kind == "batch":
        s["Hs"] = [_casida(g, k, case["dist"]) for k in _batch_orders(case)]
    elif kind == "zeig":
        s["H"] = _bse2(g, case["n"], case["dist"])
    else:
        raise ValueError(kind)
    return s


def run(state):
    kind, kw = state["case"]["kind"], state["kw"]
    if kind == "sign":
        return P.sign(state["H"], **kw)[0]
    if kind == "noalloc":
        return P.sign_noalloc(state["H"], S=state["S"], **kw)[0]
    if kind == "eig":
        D, V, _ = P.eig(state["H"], sigma=state["sigma"], **kw)
        return {"D": D, "V": V}
    if kind == "split":
        Q, A11, A22, p, _ = P.split(state["H"], **kw)
        return {"Q": Q, "A11": A11, "A22": A22, "p": p}
    if kind == "vjp":
        return P.sign_vjp_rev(state["H"], Sbar=state["G"], pos_weight=1.0, **kw)
    if kind == "casida_split":
        Q, A11, A22, _, _ = P.casida_split(state["A"], state["B"], **kw)
        return {"Q": Q, "A11": A11, "A22": A22}
    if kind == "casida_eig":
        D, V, _ = P.casida_eig(state["A"], state["B"], **kw)
        return {"D": D, "V": V}
    if kind == "batch":
        Ds, Vs, _ = P.eig_batched(state["Hs"], **kw)
        return {"D": Ds, "V": Vs}
    D, V, _ = P.zeig(state["H"], **kw)
    return {"D": D, "V": V}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Multiply-adds x 2 of the method at FP64: the front end (Cholesky with inverse and the congruence, n^3), two
    Zolotarev steps of degree 3 (the square, three factorisations with inverse and its square, the product: 5 n^3
    each), then the outputs' own products; the bytes of the inputs and outputs."""
    kind = case["kind"]
    sign = 11.0
    if kind == "batch":
        f = b = 0.0
        for k in _batch_orders(case):
            w = work({"kind": "eig", "n": 2 * k})
            f, b = f + w["flops"], b + w["bytes"]
        return {"bytes": b, "flops": f}
    if kind in ("casida_split", "casida_eig"):
        k = float(case["k"])
        if kind == "casida_split":
            return {"bytes": 8.0 * (2 + 4 + 2) * k * k, "flops": (2.0 + 12.0 + 6.0) * k ** 3}
        return {"bytes": 8.0 * (2 + 4) * k * k, "flops": (2.0 + 12.0 + 20.0) * k ** 3}
    n = float(case["n"])
    if kind in ("sign", "noalloc"):
        return {"bytes": 16.0 * n * n, "flops": (sign + 2.0) * n ** 3}
    if kind == "split":   # sketch and its orthonormal basis, projected blocks, Q
        return {"bytes": 8.0 * 2.5 * n * n, "flops": (sign + 8.0) * n ** 3}
    if kind == "vjp":     # per step two products per shifted inverse and four more, then the congruence's adjoint
        return {"bytes": 24.0 * n * n, "flops": (sign + 2.0 * (3 * 4.0 + 8.0) + 16.0) * n ** 3}
    if kind == "eig":     # split, the recursion on both halves (a quarter of a level's work per level), V, refinement
        return {"bytes": 16.0 * n * n, "flops": (sign + 8.0) * 4.0 / 3.0 * n ** 3 + 9.0 * n ** 3}
    return {"bytes": 32.0 * n * n, "flops": 4.0 * ((sign + 8.0) * 4.0 / 3.0 + 9.0) * n ** 3}   # zeig: complex products


# ---------------------------------------------------------------- the same in plain 64-bit torch
def _definite(H, sigma):
    """(L, eigenvalues, eigenvectors) of K = L^H Sigma L, Sigma H = L L^H."""
    M = sigma[:, None] * H
    L = torch.linalg.cholesky(0.5 * (M + M.mH))
    K = L.mH @ (sigma[:, None] * L)
    w, Z = torch.linalg.eigh(0.5 * (K + K.mH))
    return L, w, Z


def _default_sigma(n):
    s = torch.ones(n, device="cuda", dtype=torch.float64)
    s[n // 2:] = -1.0
    return s


def _solve_lt(L, X):
    return torch.linalg.solve_triangular(L.mH, X, upper=True)


def _exact_sign(H):
    L, w, Z = _definite(H, _default_sigma(H.shape[0]))
    return _solve_lt(L, (Z * torch.sign(w)) @ (Z.mH @ L.mH))


def _column_signs(V):
    top = V.gather(0, V.abs().argmax(0, keepdim=True))
    return V * (top.conj() / top.abs())


def _exact_eig(H, sigma):
    """D (positive ascending, then negative by magnitude) and V with V^H Sigma V = diag(sign D)."""
    L, w, Z = _definite(H, sigma)
    V = _column_signs(_solve_lt(L, Z) * torch.sqrt(w.abs()))
    order = torch.cat([torch.nonzero(w > 0).ravel(), torch.nonzero(w <= 0).ravel().flip(0)])
    return w[order].contiguous(), V[:, order].contiguous()


def _exact_vjp(H, G, weight):
    """d(<G, sign H> + weight * sum of positive eigenvalues)/dH for pseudosymmetric H (Daleckii-Krein)."""
    n = H.shape[0]
    s = _default_sigma(n)
    L, w, Z = _definite(H, s)
    V, Vit = _solve_lt(L, Z), L @ Z                      # H V = V diag(w), V^{-T} = L Z
    sg = torch.sign(w)
    diff = w[:, None] - w[None, :]
    F = torch.where(sg[:, None] != sg[None, :], (sg[:, None] - sg[None, :]) / torch.where(diff == 0, 1.0, diff), 0.0)
    X = F * (V.T @ G @ Vit) + weight * torch.diag((w > 0).double())
    X = s[:, None] * (Vit @ X @ V.T)
    return s[:, None] * (0.5 * (X + X.T))


def _polar(C):
    """Orthogonal polar factor of C by the scaled Newton iteration."""
    X = C
    for _ in range(60):
        Y = torch.linalg.inv(X).T
        mu = math.sqrt(float(torch.linalg.norm(Y) / torch.linalg.norm(X)))
        Xn = 0.5 * (mu * X + Y / mu)
        done = float(torch.linalg.norm(Xn - X) / torch.linalg.norm(Xn)) < 1e-13
        X = Xn
        if done:
            break
    return X


def _exact_casida(A, B, kind):
    LP, LR = torch.linalg.cholesky(A + B), torch.linalg.cholesky(A - B)
    C = LP.T @ LR
    if kind == "casida_split":
        U = _polar(C)
        Hc = U.T @ C
        F = torch.linalg.cholesky(0.5 * (Hc + Hc.T))
        X, Y = _solve_lt(LP, U @ F), _solve_lt(LR, F)
        A11 = F.T @ F
        return {"Q": torch.cat([torch.cat([X + Y, X - Y], 1), torch.cat([X - Y, X + Y], 1)], 0) / 2, "A11": A11,
                "A22": -A11}
    k = C.shape[0]
    O = torch.zeros_like(C)
    w, Z = torch.linalg.eigh(torch.cat([torch.cat([O, C], 1), torch.cat([C.T, O], 1)], 0))
    w, W = w[k:], Z[k:, k:] * math.sqrt(2.0)             # C = U diag(w) W^T
    X, Y = (LR @ W) / torch.sqrt(w), _solve_lt(LR, W) * torch.sqrt(w)
    V = torch.cat([torch.cat([X + Y, X - Y], 1), torch.cat([X - Y, X + Y], 1)], 0) / 2
    return {"D": torch.cat([w, -w]), "V": _column_signs(V)}


def exact(case, seed):
    """The outputs in 64 bits; None for the split, whose bases depend on the sketch the library draws."""
    kind = case["kind"]
    if kind == "split":
        return None
    s = prepare(case, seed)
    if kind in ("sign", "noalloc"):
        return _exact_sign(s["H"])
    if kind == "eig":
        D, V = _exact_eig(s["H"], torch.from_numpy(s["sigma"]).cuda().double())
        return {"D": D, "V": V}
    if kind == "vjp":
        return _exact_vjp(s["H"], s["G"], 1.0)
    if kind in ("casida_split", "casida_eig"):
        return _exact_casida(s["A"], s["B"], kind)
    if kind == "batch":
        both = [_exact_eig(H, _default_sigma(H.shape[0])) for H in s["Hs"]]
        return {"D": [d for d, _ in both], "V": [v for _, v in both]}
    D, V = _exact_eig(s["H"], _default_sigma(case["n"]).to(torch.float64))
    return {"D": D, "V": V}
