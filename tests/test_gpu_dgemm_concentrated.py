"""FP64 products A^H G of orthonormal columns with few large entries, in different rows for different columns
(csrc/dgemm_tc.cu): they cancel to zeros, and the large entries meet small ones, but their terms are not small next
to the scales, so the digits give them.  Such columns are what the orthonormalisation of a tensor with concentrated
singular vectors works on."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U = 2.0 ** -53
K, M, N, N3 = 2048, 360, 120, 16


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


def _columns(kind):
    """Fourier slices 0 .. N3 / 2 (the first and the last real) of A and G, orthonormal against each other, and the
    tensors."""
    g = torch.Generator(device="cuda").manual_seed(11)
    h = N3 // 2 + 1
    Z = torch.complex(*torch.randn((2, h, K, M + N), generator=g, device="cuda", dtype=torch.float64))
    Z.imag[0] = 0
    Z.imag[-1] = 0
    if kind == "lognormal":
        Z = torch.linalg.qr(Z * torch.exp(1.2 * torch.randn(Z.shape, generator=g, device="cuda", dtype=torch.float64)))[0]
    elif kind == "identity":
        Z = 0.02 * Z
        Z.diagonal(dim1=1, dim2=2).add_(1.0)
        Z = torch.linalg.qr(Z)[0]
    A, G = Z[:, :, :M].contiguous(), Z[:, :, M:].contiguous()
    return A, G, torch.fft.irfft(A, n=N3, dim=0), torch.fft.irfft(G, n=N3, dim=0)


def _run(api, A, G):
    B = torch.zeros((N3, M, N), dtype=torch.float64, device="cuda")
    return api.tprod_backward(A, B, G, "fp64", need_dA=False)[1]


def _time(api, A, G):
    ms = []
    for _ in range(4):
        t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t0.record()
        _run(api, A, G)
        t1.record()
        torch.cuda.synchronize()
        ms.append(t0.elapsed_time(t1))
    return min(ms[1:])


@pytest.mark.parametrize("kind", ["lognormal", "identity"])
def test_accuracy(api, kind):
    """Per element 4.5 K u sum |a||g| (2.4 K of the digits, 2 K of the products it is compared with, the transforms),
    2-norm 20 u of the same sums (16 of the digits where the sums are only just 2^-7 of the scales, 4 of the other)."""
    hA, hG, A, G = _columns(kind)
    got = torch.fft.rfft(_run(api, A, G), dim=0)
    want, size = hA.mH @ hG, hA.abs().mT @ hG.abs()
    d = (got - want).abs()
    assert bool((d <= 4.5 * K * U * size).all())
    assert float(d.norm() / size.norm()) <= 20 * U


@pytest.mark.parametrize("kind", ["lognormal", "identity"])
def test_time(api, kind):
    """Left to FP64 multiply-adds these products take ten times as long as those of normal data."""
    normal = _time(api, *_columns("normal")[2:])
    assert _time(api, *_columns(kind)[2:]) <= 3 * normal
