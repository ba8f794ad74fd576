"""FP32 products in split TF32 with short accumulations (csrc/sgemm_tc.cu), through
the t-product and its adjoints, against 64-bit references at the edges of its
tiles (128 rows, 64 columns, 16 and 128 of K)."""
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
    if kind == "graded":  # six decades inside each row
        x *= 10.0 ** rng.uniform(-3, 3, shape)
    elif kind == "huge":
        x *= 1e15
    elif kind == "tiny":
        x *= 1e-15
    elif kind == "const":  # sums of one sign, where truncated additions show most
        x[:] = 1.0 / 3.0
    elif kind == "zeros":
        x[:, : shape[1] // 2] = 0.0
    return x


# n1, n2 (= K), n4, n3: from the size on from which the split form is taken
SHAPES = [(256, 512, 128, 16), (257, 513, 129, 17), (255, 496, 191, 16), (300, 1000, 65, 16), (300, 2000, 600, 16),
          (1000, 100, 1000, 5), (700, 301, 190, 33)]


@pytest.mark.parametrize("kind", ["normal", "graded", "huge", "tiny", "const", "zeros"])
@pytest.mark.parametrize("n1,n2,n4,n3", SHAPES)
def test_split_products(api, n1, n2, n4, n3, kind):
    """C = A * B and both adjoints (the four orders of operands) from the library's
    own transforms of the operands (test_gpu_fft.py).  With u = 2^-24, worst case
    relative to |row| |col|: 4 u from the operands (2^-23 each), 8 u from the four
    truncated additions of an accumulator, 8 u inside a run of eight readings and u
    for each of the K / 128 runs.  The inverse transform adds u sqrt(log2 n3) of the
    tube's norm over all slices, with a factor of 8."""
    rng = np.random.default_rng(n1 + 7 * n2 + n4)
    A, B = _data(kind, (n3, n1, n2), rng), _data(kind, (n3, n2, n4), rng)
    G = rng.standard_normal((n3, n1, n4))
    tA, tB, tG = (torch.from_numpy(x).cuda().float() for x in (A, B, G))
    hA, hB, hG = (api.rfft3(x).to(torch.complex128) for x in (tA, tB, tG))

    def check(got, L, Rm):
        want = torch.matmul(L, Rm)
        bound = L.norm(dim=2, keepdim=True) * Rm.norm(dim=1, keepdim=True)
        big = bound.amax()  # 1e300 squared would overflow
        tube = big * (bound / big).square().sum(dim=0, keepdim=True).mul(2).sqrt()
        u = 2.0 ** -24
        tol = u * ((20 + L.shape[2] / 128) * bound + 8 * np.sqrt(np.log2(2 * n3) + 1) * tube)
        d = (torch.fft.rfft(got.double(), dim=0) - want).abs()
        assert bool((d <= tol + 1e-44).all()), float((d / tol.clamp_min(1e-300)).max())

    check(api.tprod(tA, tB), hA, hB)
    dA, dB = api.tprod_backward(tA, tB, tG, "fp32")
    check(dA, hG, hB.mH)
    check(dB, hA.mH, hG)


def test_not_finite(api):
    """An infinity or NaN makes its row (or column) not finite and leaves the others as they are."""
    torch.manual_seed(3)
    A = torch.randn(32, 256, 600, device="cuda")
    B = torch.randn(32, 600, 300, device="cuda")
    ref = api.tprod(A, B)
    A2, B2 = A.clone(), B.clone()
    A2[3, 17, 5] = float("inf")
    B2[2, 9, 40] = float("nan")
    C = api.tprod(A2, B2)
    bad = torch.zeros(256, 300, dtype=torch.bool, device="cuda")
    bad[17, :] = True
    bad[:, 40] = True
    assert not torch.isfinite(C[:, bad]).any()
    assert torch.equal(C[:, ~bad], ref[:, ~bad])
