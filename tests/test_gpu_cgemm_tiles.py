"""FP32 products on the 32 x 32 tiles of csrc/cgemm.cu, at the edges of their tiles
and of K, in the four orders of operands, against 64-bit products."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("n1,n2,n4,n3", [
    (1, 1, 1, 2), (31, 7, 33, 3), (32, 32, 32, 4), (33, 65, 31, 5), (32, 16, 500, 2), (500, 17, 32, 3),
    (1, 300, 65, 4), (64, 1000, 64, 2), (65, 129, 63, 9), (97, 200, 95, 8)])
def test_small_products(api, n1, n2, n4, n3):
    """C = A * B and both adjoints from the library's own transforms of the operands.
    A sum of 2 K real products in any order is within 2 K u of |row| |col| (u = 2^-24),
    sqrt(2) for the two parts; the inverse transform adds u sqrt(log2 n3) of the
    tube's norm over all slices, with a factor of 8."""
    torch.manual_seed(n1 + 3 * n2 + n4)
    A, B, G = (torch.randn(n3, *s, device="cuda") for s in ((n1, n2), (n2, n4), (n1, n4)))
    hA, hB, hG = (api.rfft3(x).to(torch.complex128) for x in (A, B, G))

    def check(got, L, Rm):
        want = torch.matmul(L, Rm)
        bound = L.norm(dim=2, keepdim=True) * Rm.norm(dim=1, keepdim=True)
        tube = bound.square().sum(dim=0, keepdim=True).mul(2).sqrt()
        tol = 2.0 ** -24 * (np.sqrt(2) * (2 * L.shape[2] + 4) * bound + 8 * np.sqrt(np.log2(2 * n3) + 1) * tube)
        d = (torch.fft.rfft(got.double(), dim=0) - want).abs()
        assert bool((d <= tol).all()), float((d / tol).max())

    check(api.tprod(A, B), hA, hB)
    dA, dB = api.tprod_backward(A, B, G, "fp32")
    check(dA, hG, hB.mH)
    check(dB, hA.mH, hG)
