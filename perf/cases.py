"""Performance cases of the library: what its users have it do, through the
public entry points of paper_2504_04989_gb300.

A case is a dict of plain values; `prepare` builds the inputs and the plan a
program would keep, `run` makes one pass, `exact` gives the same outputs from
torch alone in 64 bits.  A real n1 x n2 x n3 tensor is stored (n3, n1, n2).

The factors U and V of a truncated T-SVD are unique only up to a unit phase
per Fourier slice and column, so the T-SVD cases go on to the product
U * S * V^T (denoising, compression, the completion operator), which is
unique, and return it with the singular tubes S.  Their tensors have their
spectral gap at the rank R that is asked for, as a user chooses R.
"""
import math
import random

import torch

from paper_2504_04989_gb300 import api
from paper_2504_04989_gb300.completion import FillInPlan


def listed():
    return [
        # the smallest call: a t-product of small tensors, where latency and launches are the cost
        {"name": "tprod_small_fp32", "kind": "tprod", "n1": 64, "n2": 48, "n4": 32, "n3": 16, "precision": "fp32"},
        # the large square t-product of the benchmark
        {"name": "tprod_square_fp32", "kind": "tprod", "n1": 1024, "n2": 1024, "n4": 1024, "n3": 64,
         "precision": "fp32"},
        # data tensor times a thin block on the tensor cores: one Krylov product by itself
        {"name": "tprod_thin_tf32", "kind": "tprod", "n1": 2048, "n2": 2048, "n4": 120, "n3": 128,
         "precision": "tf32"},
        # one gradient step of completion in factored form: U * W of tubal rank 20 and both gradients
        {"name": "tprod_grad_lowrank_fp32", "kind": "tprod_grad", "n1": 256, "n2": 20, "n4": 256, "n3": 100,
         "precision": "fp32"},
        # forward and backward in FP64, odd sizes
        {"name": "tprod_grad_fp64", "kind": "tprod_grad", "n1": 301, "n2": 257, "n4": 190, "n3": 31,
         "precision": "fp64"},
        # projection on a subspace and its gradients, ragged sizes
        {"name": "tproj_grad_fp32", "kind": "tproj_grad", "n1": 701, "m": 60, "n2": 515, "n3": 33,
         "precision": "fp32"},
        # T-QR of a tall tensor
        {"name": "tqr_tall_fp32", "kind": "tqr", "n1": 1000, "n2": 120, "n3": 24, "precision": "fp32"},
        # the small FP64 T-SVD of the smoke test
        {"name": "tsvd_small_fp64", "kind": "tsvd", "n1": 64, "n2": 64, "n3": 16, "R": 10, "P": 5, "q": 2,
         "decay": 0.0, "precision": "fp64"},
        # the image-like T-SVD in both precisions it is used in
        {"name": "tsvd_image_fp32", "kind": "tsvd", "n1": 512, "n2": 512, "n3": 64, "R": 50, "P": 10, "q": 4,
         "decay": 1.5, "precision": "fp32"},
        {"name": "tsvd_image_fp64", "kind": "tsvd", "n1": 512, "n2": 512, "n3": 64, "R": 50, "P": 10, "q": 4,
         "decay": 1.5, "precision": "fp64"},
        # the video-like T-SVD of the benchmark's headline: the largest call
        {"name": "tsvd_video_tf32", "kind": "tsvd", "n1": 2048, "n2": 2048, "n3": 128, "R": 100, "P": 20, "q": 3,
         "decay": 0.5, "precision": "tf32"},
        # a batch of uneven tensors in one captured graph, each followed by its product
        {"name": "tsvd_batch_uneven_fp32", "kind": "batch", "count": 24, "sizes": 7, "precision": "fp32"},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["tprod", "tprod_grad", "tproj_grad", "tqr", "tsvd", "tsvd", "batch", "completion"])
    prec2 = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "tprod":
        while True:
            c = {"kind": kind, "n1": _log_int(rng, 17, 2048), "n2": _log_int(rng, 17, 2048),
                 "n4": _log_int(rng, 17, 1024), "n3": _log_int(rng, 3, 128),
                 "precision": rng.choice(["fp32", "fp32", "fp64", "tf32", "tf32x3"])}
            cost = c["n1"] * c["n2"] * c["n4"] * c["n3"] * (40 if c["precision"] == "fp64" else 1)
            if cost < 4e10:
                return c
    if kind == "tprod_grad":
        while True:
            c = {"kind": kind, "n1": _log_int(rng, 33, 1024), "n2": _log_int(rng, 9, 512),
                 "n4": _log_int(rng, 33, 1024), "n3": _log_int(rng, 3, 128), "precision": prec2}
            if c["n1"] * c["n2"] * c["n4"] * c["n3"] * (40 if prec2 == "fp64" else 1) < 2e10:
                return c
    if kind == "tproj_grad":
        while True:
            n1 = _log_int(rng, 33, 1024)
            c = {"kind": kind, "n1": n1, "m": rng.randint(5, min(n1, 128)), "n2": _log_int(rng, 33, 1024),
                 "n3": _log_int(rng, 3, 128), "precision": prec2}
            if c["n1"] * c["m"] * c["n2"] * c["n3"] * (40 if prec2 == "fp64" else 1) < 1e10:
                return c
    if kind == "tqr":
        n2 = rng.randint(9, 160)
        return {"kind": kind, "n1": _log_int(rng, 2 * n2, 1024), "n2": n2, "n3": rng.randint(3, 40),
                "precision": prec2}
    if kind == "tsvd":
        precision = rng.choice(["fp32", "fp32", "fp64", "tf32"])
        top = {"fp32": 768, "fp64": 400, "tf32": 1400}[precision]
        n1, n2 = _log_int(rng, 48, top), _log_int(rng, 48, top)
        q = rng.randint(1, 4)
        R = rng.randint(4, min(n1, n2, 150) // 3)
        P = rng.randint(4, 12)
        decay = rng.choice([0.0, 0.5, 1.0] if precision == "tf32" else [0.0, 1.0, 1.5])
        return {"kind": kind, "n1": n1, "n2": n2, "n3": _log_int(rng, 3, 64), "R": R, "P": P, "q": q,
                "decay": decay, "precision": precision}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(3, 24), "sizes": rng.randint(100, 10 ** 6), "precision": "fp32"}
    # one fill-in iteration on an image or a short video (a third of the entries missing)
    return {"kind": "completion", "n1": rng.randint(120, 300), "n2": rng.randint(120, 300),
            "n3": rng.choice([3, 3, 10, 31]), "R": rng.randint(10, 25), "P": 10, "q": 2, "precision": "fp32"}


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _randn(shape, seed, salt, dtype):
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + salt)
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _spectrum(R, decay):
    """R leading values (1 to 0.1 for decay 0, else i^-decay), then as many again, an order below."""
    if decay == 0.0:
        lead = torch.linspace(1.0, 0.1, R, dtype=torch.float64)
        tail = torch.full((R,), 0.01, dtype=torch.float64)
    else:
        s = torch.arange(1, 2 * R + 1, dtype=torch.float64) ** -decay
        lead, tail = s[:R], 0.1 * s[R:]
    return torch.cat([lead, tail])


def _low_rank(n1, n2, n3, R, decay, seed, salt, dtype):
    """A tensor of R dominant singular values per Fourier slice, a weaker rest and noise of 1e-4 of its RMS."""
    s = _spectrum(R, decay).to("cuda", dtype)
    U = torch.fft.rfft(_randn((n3, n1, 2 * R), seed, salt + 1, dtype), dim=0) / math.sqrt(n1 * n3)
    V = torch.fft.rfft(_randn((n3, n2, 2 * R), seed, salt + 2, dtype), dim=0) / math.sqrt(n2 * n3)
    X = torch.fft.irfft(torch.matmul(U * s, V.mH), n=n3, dim=0)
    X *= 1.0 / X.std()
    X += 1e-4 * _randn(X.shape, seed, salt + 3, dtype)
    return X.contiguous()


def _batch_sizes(case):
    """The uneven batch of the library's benchmark: n1, n2 ~ U{32..512}, n3 in {8, 16, 32, 64}, rank ~ U{5..40}."""
    r = random.Random(case["sizes"])
    out = []
    for _ in range(case["count"]):
        n1, n2, n3 = r.randint(32, 512), r.randint(32, 512), r.choice([8, 16, 32, 64])
        out.append((n1, n2, n3, min(r.randint(5, 40), n1 // 2, n2 // 2)))
    return out


BATCH_P, BATCH_Q = 5, 2


def _completion_data(case, seed):
    n1, n2, n3 = case["n1"], case["n2"], case["n3"]
    X = _low_rank(n1, n2, n3, case["R"], 0.0, seed, 10, torch.float32)
    X = (128.0 + 40.0 * X).clamp(0.0, 255.0)
    g = torch.Generator(device="cuda").manual_seed(1000003 * seed + 77)
    mask = (torch.rand(X.shape, generator=g, device="cuda") >= 1.0 / 3.0).to(torch.uint8)
    return X, mask


def _inputs(case, seed):
    """The tensors of a case, as prepare and exact both see them."""
    dt, k = _dtype(case), case["kind"]
    if k in ("tprod", "tprod_grad"):
        A = _randn((case["n3"], case["n1"], case["n2"]), seed, 1, dt)
        B = _randn((case["n3"], case["n2"], case["n4"]), seed, 2, dt)
        dC = _randn((case["n3"], case["n1"], case["n4"]), seed, 3, dt) if k == "tprod_grad" else None
        return A, B, dC
    if k == "tproj_grad":
        Q = _randn((case["n3"], case["n1"], case["m"]), seed, 1, dt) / math.sqrt(case["n1"] * case["n3"])
        A = _randn((case["n3"], case["n1"], case["n2"]), seed, 2, dt)
        return Q, A, _randn(A.shape, seed, 3, dt)
    if k == "tqr":
        return (_randn((case["n3"], case["n1"], case["n2"]), seed, 1, dt),)
    if k == "tsvd":
        return (_low_rank(case["n1"], case["n2"], case["n3"], case["R"], case["decay"], seed, 0, dt),)
    if k == "batch":
        return [_low_rank(n1, n2, n3, R, 0.0, seed, 10 * i, dt) for i, (n1, n2, n3, R) in enumerate(_batch_sizes(case))]
    return _completion_data(case, seed)


def prepare(case, seed):
    k, t = case["kind"], _inputs(case, seed)
    s = {"case": case, "t": t}
    if k == "tprod_grad" or k == "tproj_grad":
        t[0].requires_grad_(True)
        t[1].requires_grad_(True)
    elif k == "tsvd":
        s["plan"] = api.RbkPlan(case["n1"], case["n2"], case["n3"], case["R"], case["P"], case["q"],
                                precision=case["precision"])
    elif k == "batch":
        sizes = _batch_sizes(case)
        s["plan"] = api.RbkBatchPlan([x[:3] for x in sizes], [x[3] for x in sizes], P=BATCH_P, q=BATCH_Q,
                                     precision=case["precision"], graph=True)
    elif k == "completion":
        s["plan"] = FillInPlan(t[0], t[1], case["R"], case["P"], case["q"], precision=case["precision"])
    return s


def run(state):
    case, t = state["case"], state["t"]
    k = case["kind"]
    if k == "tprod":
        return {"C": api.tprod(t[0], t[1], case["precision"])}
    if k == "tprod_grad":
        C = api.tprod(t[0], t[1], case["precision"])
        dA, dB = torch.autograd.grad(C, (t[0], t[1]), t[2])
        return {"C": C, "dA": dA, "dB": dB}
    if k == "tproj_grad":
        Y = api.tproj(t[0], t[1], case["precision"])
        dQ, dA = torch.autograd.grad(Y, (t[0], t[1]), t[2])
        return {"Y": Y, "dQ": dQ, "dA": dA}
    if k == "tqr":
        Q, R = api.tqr(t[0])
        return {"Q": Q, "R": R}
    if k == "tsvd":
        U, S, V, sig = state["plan"](t[0])
        out = {"S": S, "X": api.lowrank(U, S, V)}
        if case["precision"] == "fp64":  # the FP32 paths' values are FP32-accurate: S has them
            out["sigma"] = sig
        return out
    if k == "batch":
        U, S, V, _ = state["plan"](t)
        return {"S": list(S), "X": [api.lowrank(u, s, v) for u, s, v in zip(U, S, V)]}
    plan = state["plan"]
    X = plan.step(1)
    return {"X": X, "C": plan.C}


def _tsvd_work(n1, n2, n3, R, P, q, es):
    h, b = n3 // 2 + 1, R + P
    m = min((q + 1) * b, n1, n2)
    # the Krylov products, the basis, the small SVD, the outputs, the product of the factors
    flops = 8.0 * h * (n1 * n2 * (2 * m - b) + n1 * m * m + n2 * m * m / 2 + m ** 3 * 2 / 3 + (n1 + n2) * m * R +
                       n1 * n2 * R)
    return {"bytes": es * n3 * (2.0 * n1 * n2 + (n1 + n2 + 1) * R), "flops": flops}


def work(case):
    k, es = case["kind"], 8 if case["precision"] == "fp64" else 4
    if k in ("tprod", "tprod_grad"):
        n1, n2, n4, n3 = case["n1"], case["n2"], case["n4"], case["n3"]
        h = n3 // 2 + 1
        g = k == "tprod_grad"
        return {"bytes": es * n3 * ((2.0 if g else 1.0) * (n1 * n2 + n2 * n4) + (2.0 if g else 1.0) * n1 * n4),
                "flops": 8.0 * h * n1 * n2 * n4 * (3 if g else 1)}
    if k == "tproj_grad":
        n1, m, n2, n3 = case["n1"], case["m"], case["n2"], case["n3"]
        # Q^T A, Q (Q^T A); Q^T dY, Q (Q^T dY), dY (A^T Q), A (dY^T Q)
        return {"bytes": es * n3 * (2.0 * n1 * m + 4.0 * n1 * n2), "flops": 8.0 * (n3 // 2 + 1) * n1 * n2 * m * 6}
    if k == "tqr":
        n1, n2, n3 = case["n1"], case["n2"], case["n3"]
        return {"bytes": es * n3 * (2.0 * n1 * n2 + n2 * n2), "flops": 8.0 * (n3 // 2 + 1) * n1 * n2 * n2 * 2}
    if k == "batch":
        ws = [_tsvd_work(n1, n2, n3, R, BATCH_P, BATCH_Q, es) for n1, n2, n3, R in _batch_sizes(case)]
        return {"bytes": sum(w["bytes"] for w in ws), "flops": sum(w["flops"] for w in ws)}
    w = _tsvd_work(case["n1"], case["n2"], case["n3"], case["R"], case["P"], case["q"], es)
    if k == "completion":  # the data, its mask and the next iterate too
        w["bytes"] += (2.0 * es + 1) * case["n3"] * case["n1"] * case["n2"]
    return w


# ---------------------------------------------------------------------------
# the same outputs in 64 bits, from torch alone
# ---------------------------------------------------------------------------
def _philox_normals(seed, n):
    """n normals of Philox4x32-10 (counter = call, key = seed) by Box-Muller, as the entry points document."""
    calls = (n + 3) // 4
    lo = 0xFFFFFFFF
    c0 = torch.arange(calls, dtype=torch.int64, device="cuda")
    c1, c2, c3 = (torch.zeros_like(c0) for _ in range(3))
    k0, k1 = seed & lo, (seed >> 32) & lo
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & lo) ^ c1) ^ k0, p1 & lo, (((p0 >> 32) & lo) ^ c3) ^ k1, p0 & lo
        k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
    u = [(x.double() + 1.0) / 4294967296.0 for x in (c0, c1, c2, c3)]
    z = []
    for a, b in ((0, 1), (2, 3)):
        r = torch.sqrt(-2.0 * torch.log(u[a]))
        z += [r * torch.cos(2 * math.pi * u[b]), r * torch.sin(2 * math.pi * u[b])]
    return torch.stack(z, dim=1).reshape(-1)[:n]


def _tsvd_exact(X, R, P, q, seed=0):
    """S, U * S * V^T and the Fourier singular values of the block Krylov T-SVD, slice by slice in complex128."""
    X = X.double()
    n3, n1, n2 = X.shape
    b = R + P
    m = min((q + 1) * b, n1, n2)
    Om = torch.fft.rfft(_philox_normals(seed, n3 * n2 * b).reshape(n3, n2, b), dim=0)
    Xh = torch.fft.rfft(X, dim=0)
    sig, out = [], torch.empty_like(Xh)
    for k in range(Xh.shape[0]):
        A = Xh[k]
        Q = torch.linalg.qr(A @ Om[k])[0]
        last = Q
        while Q.shape[1] < m:
            W = A @ (A.mH @ last)
            for _ in range(2):
                W = W - Q @ (Q.mH @ W)
            W = torch.linalg.qr(W)[0]
            W = torch.linalg.qr(W - Q @ (Q.mH @ W))[0]
            last = W[:, :m - Q.shape[1]]
            Q = torch.cat([Q, last], dim=1)
        Q = Q[:, :m]
        C = Q.mH @ A
        lam, E = torch.linalg.eigh(C @ C.mH)
        E = E[:, -R:].flip(1)
        sig.append(lam[-R:].flip(0).clamp_min(0).sqrt())
        out[k] = (Q @ E) @ (E.mH @ C)
    sig = torch.stack(sig)
    return torch.fft.irfft(sig + 0j, n=n3, dim=0), torch.fft.irfft(out, n=n3, dim=0), sig


def _fft(X):
    return torch.fft.rfft(X.double(), dim=0)


def exact(case, seed):
    k, t = case["kind"], _inputs(case, seed)
    n3 = case.get("n3")

    def back(Xh):
        return torch.fft.irfft(Xh, n=n3, dim=0)

    if k in ("tprod", "tprod_grad"):
        A, B = _fft(t[0]), _fft(t[1])
        out = {"C": back(A @ B)}
        if k == "tprod_grad":
            G = _fft(t[2])
            out["dA"], out["dB"] = back(G @ B.mH), back(A.mH @ G)
        return out
    if k == "tproj_grad":
        Q, A, G = (_fft(x) for x in t)
        return {"Y": back(Q @ (Q.mH @ A)), "dQ": back(G @ (A.mH @ Q) + A @ (G.mH @ Q)), "dA": back(Q @ (Q.mH @ G))}
    if k == "tqr":
        Q, R = torch.linalg.qr(_fft(t[0]))
        d = torch.diagonal(R, dim1=1, dim2=2)
        d = d / d.abs()
        return {"Q": back(Q * d[:, None, :]), "R": back(R * d.conj()[:, :, None])}
    if k == "tsvd":
        S, X, sig = _tsvd_exact(t[0], case["R"], case["P"], case["q"])
        out = {"S": S, "X": X}
        if case["precision"] == "fp64":
            out["sigma"] = sig
        return out
    if k == "batch":
        got = [_tsvd_exact(x, sz[3], BATCH_P, BATCH_Q, seed=i) for i, (x, sz) in enumerate(zip(t, _batch_sizes(case)))]
        return {"S": [g[0] for g in got], "X": [g[1] for g in got]}
    M, mask = t[0].double(), t[1].bool()
    _, X, _ = _tsvd_exact(M * mask, case["R"], case["P"], case["q"])
    return {"X": X, "C": torch.where(mask, M, X)}
