"""GPU mode-3 transforms at the lengths where their kernels change: powers of two
in registers (and the two-thread form of FP64 n3 = 128), folded direct products
of odd and even n3, mixed-radix passes, with planes around the tile sizes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LENGTHS = [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 14, 16, 31, 32, 33, 64, 75, 96, 100, 127, 128, 130, 150, 159, 160, 161]


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("n3", LENGTHS)
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_transforms(api, n3, precision):
    """Every Fourier slice (and every frontal slice of the inverse) against the
    64-bit transform, 2-norm.  A transform's rounding grows as u sqrt(log2 n)
    (random signs) for the radix forms and stays below that for runs of 8; the
    bound leaves a factor of 8 (u the unit roundoff)."""
    dt, u = (torch.float32, 2.0 ** -24) if precision == "fp32" else (torch.float64, 2.0 ** -53)
    tol = 8 * u * np.sqrt(np.log2(2 * n3) + 1)
    for plane in ((1, 1), (3, 11), (31, 33), (64, 129)):
        rng = np.random.default_rng(1000 * n3 + plane[1])
        X = torch.from_numpy(rng.standard_normal((n3,) + plane)).to("cuda", dt)
        Xh = api.rfft3(X)
        ref = torch.fft.rfft(X.double(), dim=0)
        assert float(Xh[0].imag.abs().max()) == 0.0
        if n3 % 2 == 0:
            assert float(Xh[-1].imag.abs().max()) == 0.0
        d = (Xh.to(torch.complex128) - ref).flatten(1).norm(dim=1)
        # a slice of few values can be small by chance: scale by the tensor's own
        scale = float(ref.norm()) / np.sqrt(len(ref))
        assert float(d.max()) <= tol * scale, (plane, float(d.max()) / scale, tol)
        back = api.irfft3(ref.to(Xh.dtype), n3)
        ref2 = torch.fft.irfft(ref.to(Xh.dtype).to(torch.complex128), n=n3, dim=0)
        d = (back.double() - ref2).flatten(1).norm(dim=1)
        scale = float(ref2.norm()) / np.sqrt(n3)
        assert float(d.max()) <= tol * scale, (plane, float(d.max()) / scale, tol)
