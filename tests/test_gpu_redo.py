"""Elements that the tensor-core products leave to the direct sums behind them
(csrc/tc_redo.cuh): infinities and NaN in either operand and all four orders of
operands, at ragged sizes."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("many", [False, True])  # from the list of marks; by tiles, where it does not hold them
@pytest.mark.parametrize("n1,n2,n4", [(300, 517, 259), (1025, 1000, 67)])
def test_infinities(api, precision, n1, n2, n4, many):
    """Two slices, the sums and differences of the two real ones (n3 = 2), so C, dA and dB come from real
    products: infinities and NaN where those of the spectra have them, and every element that meets none
    to the bit what the product without them gives."""
    dt = torch.float64 if precision == "fp64" else torch.float32
    inf, nan = float("inf"), float("nan")
    g = torch.Generator(device="cuda").manual_seed(n1)
    A, B, G = (torch.randn((2,) + s, generator=g, device="cuda", dtype=dt) for s in ((n1, n2), (n2, n4), (n1, n4)))

    def spoil(X, r0):
        Y = X.clone()
        Y[0, r0, 5], Y[0, r0, 9], Y[1, -1, -1] = inf, -inf, -inf
        Y[0, 40, 3] = nan
        if many:
            Y[1, 1::2, 7] = inf
        return Y

    def check(got, clean, L, R):
        hL, hR = (api.rfft3(x.contiguous()).real.double() for x in (L, R))
        want = torch.matmul(hL, hR)
        want = api.irfft3(torch.complex(want, torch.zeros_like(want)), 2)
        rows, cols = (~torch.isfinite(L)).any(dim=2).any(dim=0), (~torch.isfinite(R)).any(dim=1).any(dim=0)
        bad = rows[:, None] | cols[None, :]
        assert torch.equal(torch.isnan(got[:, bad]), torch.isnan(want[:, bad]))
        infinite = torch.isinf(want)
        assert bool(infinite.any()) and torch.equal(got[infinite], want[infinite].to(dt))
        assert torch.equal(got[:, ~bad], clean[:, ~bad])

    A2, B2, G2 = spoil(A, 17), spoil(B, 2), spoil(G, 31)
    check(api.tprod(A2, B, precision), api.tprod(A, B, precision), A2, B)
    if not many:
        check(api.tprod(A, B2, precision), api.tprod(A, B, precision), A, B2)
    dA, dB = api.tprod_backward(A, B, G, precision)
    dA2, dB2 = api.tprod_backward(A, B, G2, precision)
    check(dA2, dA, G2, B.mT)
    if not many:
        check(dB2, dB, A.mT, G2)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_nothing_finite(api, precision):
    """Every element marked: a tensor full of NaN gives one."""
    dt = torch.float64 if precision == "fp64" else torch.float32
    A = torch.full((4, 300, 400), float("nan"), dtype=dt, device="cuda")
    B = torch.randn(4, 400, 200, dtype=dt, device="cuda")
    assert bool(torch.isnan(api.tprod(A, B, precision)).all())
