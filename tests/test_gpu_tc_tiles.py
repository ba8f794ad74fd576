"""Tensor-core t-products (csrc/tc_gemm.cu) in TF32, BF16 and split TF32 on integers,
whose products and sums are exact in every mode: at the edges of the tiles (128 rows,
128 and 256 columns) and of the stages of K, and with several tiles per CTA; and T-SVDs whose blocks
have even and odd numbers of columns (16-byte and 4-byte rows of the split copies)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("precision", ["tf32", "bf16", "tf32x3"])
@pytest.mark.parametrize("n1,n2,n4,n3", [
    (1, 1, 1, 1), (128, 16, 64, 2), (127, 15, 63, 1), (129, 33, 65, 2), (130, 8, 128, 1), (300, 100, 129, 2),
    (257, 40, 200, 1), (40001, 24, 130, 2), (20000, 50, 60, 2), (5000, 7, 700, 1)])
def test_exact_on_integers(api, n1, n2, n4, n3, precision):
    """|entries| <= 4 and n3 <= 2: transforms within 8, sums within 64 * 2 * 100 * 2 < 2^24, no rounding."""
    torch.manual_seed(n1 + n2 + n4)
    A = torch.randint(-4, 5, (n3, n1, n2), device="cuda").float()
    B = torch.randint(-4, 5, (n3, n2, n4), device="cuda").float()
    got = api.tprod(A, B, precision=precision)
    hA, hB = torch.fft.rfft(A.double(), dim=0), torch.fft.rfft(B.double(), dim=0)
    want = torch.fft.irfft(hA @ hB, n=n3, dim=0).round().float()
    assert torch.equal(got, want)


@pytest.mark.parametrize("R,P", [(10, 3), (10, 4), (11, 4), (12, 4), (1, 0)])
def test_blocks(api, R, P):
    """Singular values of the tensor-core orthonormalisation (n1 >= 1024) against the FP64 path's at
    the T-SVD parity bar."""
    torch.manual_seed(R + P)
    A = torch.randn(3, 1030, 60, device="cuda")
    om = torch.randn(3, 60, R + P, device="cuda")
    a = api.rbk(A, R, P, 2, precision="fp32", omega=om)[3]
    b = api.rbk(A.double(), R, P, 2, precision="fp64", omega=om.double())[3]
    assert float(((a - b).abs() / b).max()) < 1e-4
