"""Eigenvalues and eigenvectors of the small SVD (csrc/eig.cu): the bisection's last
rounds on graded spectra, and the back-transformation by pairs of reflectors at even
and odd m, around its warps' slots of 32 entries and its CTAs' numbers of vectors,
through T-SVDs whose basis is the whole space (m = n)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


def _full_basis(api, A, R, precision):
    n = A.shape[1]
    P = min(n, 128) - R
    return api.rbk(A, R, P, -(-n // (R + P)) - 1, precision=precision)


@pytest.mark.parametrize("n,n3,R", [(1, 2, 1), (2, 3, 1), (3, 5, 2), (4, 1, 4), (31, 4, 5), (32, 9, 17), (33, 3, 16), (64, 60, 21),
                                    (65, 20, 33), (127, 6, 50), (128, 40, 7), (300, 33, 50), (481, 2, 100), (512, 5, 3)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp32", 1e-4)])
def test_vectors(api, n, n3, R, precision, tol):
    """A * V = U * S and U^T * U = V^T * V = I per frontal slice, at the T-SVD's parity
    bars over a spectrum that keeps within a factor of ten (diagonal plus noise)."""
    torch.manual_seed(n + R)
    A = torch.randn(n3, n, n, dtype=torch.float64, device="cuda") * 0.1 / n ** 0.5
    A[0] += torch.diag(torch.linspace(2.0, 1.0, n, dtype=torch.float64, device="cuda"))
    A = A if precision == "fp64" else A.float()
    U, S, V, sig = _full_basis(api, A, R, precision)
    hA, hU, hV = (torch.fft.rfft(x.double(), dim=0) for x in (A, U, V))
    sig = sig[:hA.shape[0]]
    eye = torch.eye(R, dtype=hU.dtype, device="cuda")
    assert float((hA @ hV - hU * sig[:, None, :]).abs().max()) < tol * float(sig.max())
    assert float((hU.mH @ hU - eye).abs().max()) < tol
    assert float((hV.mH @ hV - eye).abs().max()) < tol


@pytest.mark.parametrize("n,decades", [(5, 3), (64, 6), (200, 7), (300, 1), (128, 12)])
def test_graded_fp64(api, n, decades):
    """sigma^2 within 16 n eps sigma_1^2 (the eigenvalues of a Gram matrix rounded entry by entry),
    over spectra of several decades, and equal ones (a cluster)."""
    torch.manual_seed(n)
    q1, q2 = (torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda"))[0] for _ in range(2))
    s = 10.0 ** torch.linspace(0, -decades, n, dtype=torch.float64, device="cuda")
    s[n // 2:] = s[n // 2]
    R = min(n, 100)
    sig = _full_basis(api, ((q1 * s) @ q2)[None].contiguous(), R, "fp64")[3]
    want = torch.linalg.svdvals((q1 * s) @ q2)[:R]
    assert float((sig[0].square() - want.square()).abs().max()) < 16 * n * 2.0 ** -52
