"""Products with more rows or columns than 65535 blocks of 32 (the limit of a
grid's second dimension), in both precisions and both operands."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


@pytest.mark.parametrize("precision,k", [("fp64", 16), ("fp32", 64)])
@pytest.mark.parametrize("wide", [False, True])
def test_tall(api, precision, k, wide):
    """65536 blocks and a row more; one slice in the transform (n3 = 1), so the result is the plain
    product: |d| <= 2 K u |row| |col|, the bound of a dot product of K terms twice over."""
    n = 65536 * 32 + 1
    dt = torch.float64 if precision == "fp64" else torch.float32
    u = 2.0 ** (-53 if precision == "fp64" else -24)
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn((1, n, k), generator=g, device="cuda", dtype=dt)
    B = torch.randn((1, k, k), generator=g, device="cuda", dtype=dt)
    if wide:  # C^T = B^T A^T
        C = api.tprod(B.mT.contiguous(), A.mT.contiguous(), precision)[0].T
    else:
        C = api.tprod(A, B, precision)[0]
    bad = 0
    for r in range(0, n, 1 << 18):
        a = A[0, r:r + (1 << 18)]
        d = (C[r:r + (1 << 18)].double() - a.double() @ B[0].double()).abs()
        bad += int((d > 2 * k * u * a.double().norm(dim=1, keepdim=True) * B[0].double().norm(dim=0)).sum())
    assert bad == 0
