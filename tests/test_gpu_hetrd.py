"""The tridiagonalisation of the small SVD (csrc/eig.cu) at sizes around its warps,
strips, clusters and memory layouts, through T-SVDs whose basis is the whole
space (m = n): singular values against a 64-bit SVD, and bitwise equal reruns."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# n = m and n3 (h = n3 // 2 + 1 slices): clusters of 8, 4, 2 and 1 CTAs, rows in shared memory (partials
# there or in L2) and in L2
SIZES = [(1, 1), (2, 3), (3, 2), (7, 4), (31, 5), (33, 40), (40, 30), (64, 31), (65, 75), (100, 160), (129, 29),
         (160, 28), (200, 33), (257, 9), (300, 16), (300, 64), (300, 76), (401, 20), (512, 3), (511, 31)]


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("n,n3", SIZES)
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
def test_full_basis(api, n, n3, precision, tol):
    """At the T-SVD parity bars for singular values (1e-10 FP64, 1e-4 FP32)."""
    torch.manual_seed(n + n3)
    A = torch.randn(n3, n, n, dtype=torch.float64, device="cuda")
    if precision == "fp32":
        A = A.float()
    R = max(1, min(n // 3, 100))
    P = min(n, 128) - R
    q = -(-n // (R + P)) - 1
    out = api.rbk(A, R, P, q, precision=precision, return_info=True)
    assert out[4]["status"] == 0 and out[4]["m_eff"] == n
    want = torch.linalg.svdvals(torch.fft.rfft(A.double(), dim=0))[:, :R]
    assert float(((out[3] - want).abs() / want).max()) < tol
    again = api.rbk(A, R, P, q, precision=precision)
    assert all(torch.equal(x, y) for x, y in zip(out[:4], again))
