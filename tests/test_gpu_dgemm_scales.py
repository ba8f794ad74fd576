"""FP64 products on data whose scales are uneven along K (csrc/dgemm_tc.cu): the
accuracy of FP64 multiply-adds whatever the scales.  Operands are fixed-point numbers
of 51 bits times powers of two, so the exact product comes from nine exact partial ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U = 2.0 ** -53


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


def _fixed(shape, g):
    """Three slices of 17 bits with signs: X = s0 + s1 2^-17 + s2 2^-34, and X (48 .. 51 bits)."""
    s = [torch.randint(-(1 << 16), 1 << 16, shape, generator=g, device="cuda").double() for _ in range(3)]
    return s, s[0] + s[1] * 2.0 ** -17 + s[2] * 2.0 ** -34


def _exact(sa, sb):
    """sum_st A_s B_t 2^-17(s+t): each product exact (16 + 16 bits and K <= 2^20 terms), the nine added in long double."""
    out = 0
    for s in range(3):
        for t in range(3):
            p = torch.matmul(sa[s], sb[t]).cpu().numpy().astype(np.longdouble)
            out = out + p * np.longdouble(2.0) ** (-17 * (s + t))
    return out


def _scales(kind, m, k, n, g):
    """Row scales, K scales of A and of B (exponents of two) and what is zero in either."""
    def rnd(size, bits):
        return torch.randint(-bits, bits + 1, (size,), generator=g, device="cuda")
    z = torch.zeros(k, dtype=torch.int64, device="cuda")
    za = torch.ones((m, k), dtype=torch.float64, device="cuda")
    zb = torch.ones((k, n), dtype=torch.float64, device="cuda")
    ea, eb = z[None, :].repeat(m, 1), z[:, None].repeat(1, n)
    if kind.startswith("opposed"):
        d = rnd(k, int(kind[7:]) // 2)
        ea, eb = ea + d[None, :], eb - d[:, None]
    elif kind == "rows":  # and rows and columns of any size
        d = rnd(k, 20)
        ea, eb = ea + d[None, :] + rnd(m, 100)[:, None], eb - d[:, None] + rnd(n, 100)[None, :]
    elif kind == "sentinel":  # large entries of A that meet zeros: one of a row, a whole column
        ea[m // 2, k // 3] = 60
        ea[:, k // 2] = 60
        zb[k // 3] = 0
        zb[k // 2] = 0
    elif kind == "half":  # a column of large entries that meet zeros in half of B's columns
        ea[:, k // 2] = 60
        zb[k // 2, ::2] = 0
    elif kind == "outlier":  # large entries that count: their row and column, and the others
        ea[m // 2, k // 3] = 40
        eb[k // 2, n // 2] = 40
    elif kind == "blocks":  # zeros against entries
        za[: m // 2, k // 2:] = 0
        za[m // 2:, : k // 2] = 0
        zb[: k // 2, n // 2:] = 0
        zb[k // 2:, : n // 2] = 0
        d = rnd(k, 20)
        ea, eb = ea + d[None, :], eb - d[:, None]
    elif kind == "triangular":  # W R^-1: columns of W and rows of the upper triangular R^-1 in opposed scales
        d = -2 * torch.arange(k, device="cuda") // 3
        ea, eb = ea + d[None, :], eb - d[:, None]
        zb = zb.triu()
    return ea, eb, za, zb


KINDS = ["opposed0", "opposed10", "opposed20", "opposed40", "opposed120", "rows", "sentinel", "half", "outlier", "blocks",
         "triangular"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("m,k,n", [(130, 256, 520), (501, 70, 333)])
@pytest.mark.parametrize("order", ["NN", "NH", "HN"])
def test_scales(api, order, m, k, n, kind):
    """n3 = 1 (the transform leaves the one slice as it is): C = A B, dA = G B^T and dB = A^T G.  Per element within
    max(2.4 K, 74) u sum |a||b|, the worst case of FP64 multiply-adds over the 2 K parts and a fifth more; per product, 2-norm,
    4 u (FP64 multiply-adds: 2.5 u on such data).  Where every term is zero the result is."""
    g = torch.Generator(device="cuda").manual_seed(m + 3 * n)
    sa, A = _fixed((m, k), g)
    sb, B = _fixed((k, n), g)
    ea, eb, za, zb = _scales(kind, m, k, n, g)
    ra, rb = ea.amax(dim=1, keepdim=True), eb.amax(dim=0, keepdim=True)
    pa, pb = za * 2.0 ** ea.double(), zb * 2.0 ** eb.double()
    A, B = A * pa, B * pb
    if kind.startswith("opposed") or kind in ("rows", "triangular", "blocks"):
        # the scales along K cancel, those of rows and columns come out
        dr, dc = ea[:, :1] - ea[:1, :1], eb[:1, :] - eb[:1, :1]
        off = (ea[0, 0] + eb[0, 0]).double()
        want = _exact([x * za for x in sa], [x * zb for x in sb])
        want = want * (2.0 ** (dr.double() + dc.double() + off)).cpu().numpy()
    else:  # the large entries apart: powers of two, in products of their own
        big = (ea > 0)
        colA, rowB = big.any(dim=0) | (eb > 0).any(dim=1), None
        want = _exact([x * za * ~colA for x in sa], [x * zb * ~colA[:, None] for x in sb])
        for q in torch.nonzero(colA)[:, 0].tolist():
            a = A[:, q].cpu().numpy().astype(np.longdouble)
            b = B[q].cpu().numpy().astype(np.longdouble)
            want = want + np.outer(a, b)
    if order == "NN":
        got = api.tprod(A[None], B[None], "fp64")[0]
    elif order == "NH":  # G = A, B^T stored
        got = api.tprod_backward(torch.zeros((1, m, n), dtype=torch.float64, device="cuda"), B.T.contiguous()[None], A[None],
                                 "fp64", need_dB=False)[0][0]
    else:
        got = api.tprod_backward(A.T.contiguous()[None], torch.zeros((1, m, n), dtype=torch.float64, device="cuda"), B[None],
                                 "fp64", need_dA=False)[1][0]
    size = torch.matmul(A.abs(), B.abs()).cpu().numpy()
    d = np.abs((got.cpu().numpy() - want).astype(np.float64))
    assert (d <= max(2.4 * k, 74) * U * size).all(), float((d / np.maximum(size, 1e-300)).max() / U)
    # row by row, so that large rows do not hide small ones
    w = want.astype(np.float64)
    rel = np.linalg.norm(d / np.abs(w).max(axis=1, keepdims=True).clip(1e-300), axis=1)
    rel /= np.linalg.norm(w / np.abs(w).max(axis=1, keepdims=True).clip(1e-300), axis=1).clip(1e-300)
    if kind not in ("outlier", "rows"):  # there a row's norm is that of its largest column
        assert rel.max() <= 4 * U, rel.max() / U


def test_update_of_marked_elements(api):
    """dQ = dY (A^T Q) + A (dY^T Q) adds a product to what is there: on entries that meet zeros and large
    columns, against the same formula of torch, with 64 u sum |.||.| (three products of K <= 600 terms)."""
    g = torch.Generator(device="cuda").manual_seed(4)
    Q = torch.randn((2, 600, 90), generator=g, device="cuda", dtype=torch.float64)
    A, Y = (torch.randn((2, 600, 500), generator=g, device="cuda", dtype=torch.float64) for _ in range(2))
    A[:, :300, 250:] = 0
    Y[:, 300:, :250] = 0
    A[:, :, 7] *= 1e12
    Y[:, :, 9] *= 1e-9
    dQ, dA = api.tproj_backward(Q, A, Y, "fp64")
    hQ, hA, hY = (torch.stack([x[0] + x[1], x[0] - x[1]]) for x in (Q, A, Y))

    def back(h):
        return torch.stack([h[0] + h[1], h[0] - h[1]]) / 2

    want = back(hY @ (hA.mT @ hQ) + hA @ (hY.mT @ hQ))
    size = back(hY.abs() @ (hA.abs().mT @ hQ.abs()) + hA.abs() @ (hY.abs().mT @ hQ.abs())).abs().amax(dim=0)
    assert bool(((dQ - want).abs() <= 64 * U * size).all())
    want = back(hQ @ (hQ.mT @ hY))
    size = back(hQ.abs() @ (hQ.abs().mT @ hY.abs())).abs().amax(dim=0)
    assert bool(((dA - want).abs() <= 64 * U * size).all())
