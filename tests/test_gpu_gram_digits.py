"""The exact Gram of the FP32 small SVD in base-256 digits on the tensor cores
(csrc/gram_int.cu) is the 64-bit integer kernel's to the bit, so the whole T-SVD is:
at the edges of its tiles (32 and 64 columns of the basis), of a stage (64 rows of
C^H) and of an accumulation (320 rows), and beyond 4096 rows."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("n1,n2,n3,b,q", [  # m = min(b (q + 1), n1, n2)
    (40, 63, 3, 1, 0), (40, 64, 2, 8, 3), (70, 65, 3, 11, 2), (90, 319, 2, 16, 3), (90, 320, 4, 13, 4),
    (200, 321, 3, 43, 2), (150, 641, 2, 32, 3), (600, 1000, 1, 128, 3), (30, 4097, 2, 6, 3), (24, 9001, 1, 12, 1)])
@pytest.mark.parametrize("kind", ["normal", "one_sign"])
def test_equals_integer_gram(api, n1, n2, n3, b, q, kind):
    torch.manual_seed(n1 + n2)
    A = torch.randn(n3, n1, n2, device="cuda")
    if kind == "one_sign":  # a column of C^H of nearly equal entries: the largest digit sums
        A = 1.0 + 1e-3 * A
    R = max(1, b - 2)
    x = api.rbk(A, R, b - R, q, precision="fp32", seed=5)
    y = api.rbk(A, R, b - R, q, precision="fp32", seed=5, gram_int=True)
    for u, v in zip(x, y):
        assert torch.equal(u, v)
