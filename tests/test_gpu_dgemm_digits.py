"""FP64 products as digit products on the tensor cores (csrc/dgemm_tc.cu), through
the t-product and its adjoints, against 64-bit references at the edges of its
tiles (128 rows, 32 columns, 32 and 192 of K) and on data that stress the digits."""
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


def _data(kind, shape, rng):
    x = rng.standard_normal(shape)
    if kind == "graded":  # twelve decades inside each row
        x *= 10.0 ** rng.uniform(-6, 6, shape)
    elif kind == "huge":
        x *= 1e150
    elif kind == "tiny":
        x *= 1e-150
    elif kind == "const":  # every digit the same in every term: the largest digit sums
        x[:] = 0.50196078431372548  # 0x0.80808080...
    elif kind == "zeros":
        x[:, : shape[1] // 2] = 0.0
    return x


# n1, n2 (= K), n4, n3: all above the size from which the digit form is taken
SHAPES = [(128, 256, 32, 16), (129, 257, 33, 17), (127, 96, 97, 16), (300, 1000, 31, 4), (1, 2000, 500, 9),
          (640, 16, 640, 3), (257, 301, 190, 5)]


@pytest.mark.parametrize("kind", ["normal", "graded", "huge", "tiny", "const", "zeros"])
@pytest.mark.parametrize("n1,n2,n4,n3", SHAPES)
def test_digit_products(api, n1, n2, n4, n3, kind):
    """C = A * B and both adjoints (the four orders of operands) from the library's
    own transforms of the operands (test_gpu_fft.py).  Per Fourier slice the digit
    form rounds each operand to 2^-56 of its row's scale and the result once: below
    8 u sqrt(2 K) |row| |col| of that slice (u = 2^-53).  The inverse transform adds
    u sqrt(log2 n3) of the tube's norm over all slices, with the same factor of 8."""
    rng = np.random.default_rng(n1 + 7 * n2 + n4)
    A, B = _data(kind, (n3, n1, n2), rng), _data(kind, (n3, n2, n4), rng)
    G = rng.standard_normal((n3, n1, n4))
    tA, tB, tG = (torch.from_numpy(x).cuda() for x in (A, B, G))
    hA, hB, hG = (api.rfft3(x) for x in (tA, tB, tG))

    def check(got, L, Rm):
        want = torch.matmul(L, Rm)
        bound = L.norm(dim=2, keepdim=True) * Rm.norm(dim=1, keepdim=True)
        big = bound.amax()  # 1e300 squared would overflow
        tube = big * (bound / big).square().sum(dim=0, keepdim=True).mul(2).sqrt()
        u = 2.0 ** -53
        tol = 8 * u * (np.sqrt(2 * L.shape[2]) * bound + np.sqrt(np.log2(2 * n3) + 1) * tube)
        d = (torch.fft.rfft(got, dim=0) - want).abs()
        assert bool((d <= tol + 1e-320).all()), float((d / tol.clamp_min(1e-300)).max())

    check(api.tprod(tA, tB), hA, hB)
    dA, dB = api.tprod_backward(tA, tB, tG, "fp64")
    check(dA, hG, hB.mH)
    check(dB, hA.mH, hG)


def test_not_finite(api):
    """An infinity or NaN makes its row (or column) not finite and leaves the others as they are."""
    torch.manual_seed(3)
    A = torch.randn(8, 256, 300, dtype=torch.float64, device="cuda")
    B = torch.randn(8, 300, 100, dtype=torch.float64, device="cuda")
    ref = api.tprod(A, B)
    A2, B2 = A.clone(), B.clone()
    A2[3, 17, 5] = float("inf")
    B2[2, 9, 40] = float("nan")
    C = api.tprod(A2, B2)
    bad = torch.zeros(256, 100, dtype=torch.bool, device="cuda")
    bad[17, :] = True
    bad[:, 40] = True
    assert not torch.isfinite(C[:, bad]).any()
    assert torch.equal(C[:, ~bad], ref[:, ~bad])
