"""FP32 products in exact BF16 parts (csrc/sgemm_tc.cu): the rounding of FP32
multiply-adds or less for short sums, and the lower end of FP32's range."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

U = 2.0 ** -24


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("k", [20, 32, 33, 48, 61])
def test_short_sums(api, k, positive):
    """n3 = 1 (the transform leaves the one slice as it is).  Expected, 2-norm: a truncated sum per 16 complex terms and
    the additions behind, 1.1 to 1.2 u of the result; FP32 multiply-adds 1.4 u (K = 20) to 2.3 u (61).  Bound: 1.5 u."""
    g = torch.Generator(device="cuda").manual_seed(k)
    A = torch.randn((1, 2048, k), generator=g, device="cuda")
    B = torch.randn((1, k, 2048), generator=g, device="cuda")
    if positive:
        A, B = A.abs(), B.abs()
    want = A[0].double() @ B[0].double()
    d = api.tprod(A, B, "fp32")[0].double() - want
    assert float(d.norm() / want.norm()) <= 1.5 * U


@pytest.mark.parametrize("order", ["NN", "NH", "HN"])
@pytest.mark.parametrize("kind", ["products", "subnormal", "tails", "opposed", "rows"])
def test_small_values(api, kind, order):
    """Entries and products near 2^-126: 4 K u sum |a||b| and a subnormal's half unit for each of the 2 K terms."""
    m, k, n = 390, 300, 777
    g = torch.Generator(device="cuda").manual_seed(11)
    A = torch.randn((m, k), generator=g, device="cuda")
    B = torch.randn((k, n), generator=g, device="cuda")
    if kind == "products":
        A, B = A * 1e-22, B * 1e-15
    elif kind == "subnormal":
        A, B = A * 1e-39, B * 1e12
    elif kind == "tails":  # most of A's columns far below its others, which meet small rows of B
        A[:, 3:] *= 1e-37
        B[:3] *= 1e-36
    elif kind == "opposed":
        A, B = A * 1e-33, B * 1e30
        A[:, ::2] *= 1e30
        B[::2] *= 1e-30
    else:  # a few rows of A and columns of B
        A[5], A[200] = A[5] * 1e-36, 0.0
        B[:, 9], B[:, 700] = B[:, 9] * 1e-38, 0.0
    size = A.double().abs() @ B.double().abs()
    want = A.double() @ B.double()
    zero = torch.zeros((1, m, n), device="cuda")
    if order == "NN":
        got = api.tprod(A[None], B[None], "fp32")[0]
    elif order == "NH":
        got = api.tprod_backward(zero, B.T.contiguous()[None], A[None], "fp32", need_dB=False)[0][0]
    else:
        got = api.tprod_backward(A.T.contiguous()[None], zero, B[None], "fp32", need_dA=False)[1][0]
    assert bool(((got.double() - want).abs() <= 4 * k * U * size + 2 * k * 2.0 ** -150).all())
