"""The panel Cholesky + inverse of the block orthonormalisation (csrc/cholqr.cu)
through the T-QR, at block widths around its panels (8 rows), tiles (4) and
launch sizes (80, 120, 128), with and without dependent columns."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

WIDTHS = [1, 2, 7, 8, 9, 15, 16, 17, 31, 33, 60, 79, 80, 81, 88, 119, 120, 121, 127, 128]


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("n2", WIDTHS)
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_tqr_widths(api, n2, precision):
    """Q and R of a well-conditioned tall tensor, unique with diag(R_k) >= 0, at
    the T-QR parity bars (1e-10 FP64, 2e-4 FP32; condition numbers below 30)."""
    dt, tol = (torch.float64, 1e-10) if precision == "fp64" else (torch.float32, 2e-4)
    torch.manual_seed(n2)
    A = torch.randn(5, n2 + 50, n2, dtype=torch.float64, device="cuda").to(dt)
    Q, R, info = api.tqr(A, return_info=True)
    assert info["status"] == 0 and info["dead_columns"] == 0
    q, r = torch.linalg.qr(torch.fft.rfft(A.double(), dim=0))
    d = torch.diagonal(r, dim1=1, dim2=2)
    d = d / d.abs()
    want = torch.fft.irfft(q * d[:, None, :], n=5, dim=0)
    assert float((Q.double() - want).abs().max()) < tol * float(want.abs().max())
    want = torch.fft.irfft(r * d.conj()[:, :, None], n=5, dim=0)
    assert float((R.double() - want).abs().max()) < tol * float(want.abs().max())


@pytest.mark.parametrize("n2", [2, 8, 9, 17, 60, 120, 121, 128])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_tqr_dependent_columns(api, n2, precision):
    """The first column again in the last place (rounding may leave it a direction of
    its own) and a zero column (always found and replaced): Q keeps orthonormal
    columns and Q * R is the tensor."""
    dt, tol = (torch.float64, 1e-10) if precision == "fp64" else (torch.float32, 2e-4)
    torch.manual_seed(n2)
    A = torch.randn(5, n2 + 50, n2, dtype=torch.float64, device="cuda").to(dt)
    A[:, :, -1] = A[:, :, 0]
    if n2 > 8:
        A[:, :, n2 // 2] = 0.0
    Q, R, info = api.tqr(A, return_info=True)
    assert info["dead_columns"] >= (3 if n2 > 8 else 0)  # on each of the 3 Fourier slices
    q = torch.fft.rfft(Q.double(), dim=0)
    eye = torch.eye(n2, dtype=q.dtype, device="cuda")
    assert float((q.mH @ q - eye).abs().max()) < tol
    back = torch.fft.irfft(q @ torch.fft.rfft(R.double(), dim=0), n=5, dim=0)
    assert float((back - A.double()).abs().max()) < tol * float(A.abs().max()) * n2 ** 0.5
