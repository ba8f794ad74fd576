"""info->status of a T-SVD whose tensor-core products give up: the waits of their
pipelines are let run out at once (TSVD_FLAG_EXPIRE), and the call ends and says so."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIMT, EXPIRE = 4, 64  # TSVD_FLAG_SIMT, TSVD_FLAG_EXPIRE


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import _lib
    return _lib


def _status(lib, precision, flags, n=384, n3=16, R=50, P=10, q=1):
    dt = torch.float64 if precision == "fp64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(9)
    A = torch.randn((n3, n, n), generator=g, device="cuda", dtype=dt)
    p = lib.TsvdParams(R=R, P=P, q=q, precision=lib.PRECISIONS[precision], seed=1, flags=flags)
    nbytes = C.c_size_t()
    lb = lib.load()
    assert lb.tsvd_rbk_workspace_size(n, n, n3, C.byref(p), C.byref(nbytes)) == 0
    ws = torch.empty(nbytes.value, dtype=torch.uint8, device="cuda")
    U, V = (torch.empty((n3, n, R), dtype=dt, device="cuda") for _ in range(2))
    S = torch.empty((n3, R), dtype=dt, device="cuda")
    sig = torch.empty((n3 // 2 + 1, R), dtype=torch.float64, device="cuda")
    info = lib.TsvdInfo()
    s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    rc = lb.tsvd_rbk(C.c_void_p(A.data_ptr()), n, n, n3, C.byref(p), None, C.c_void_p(U.data_ptr()), C.c_void_p(S.data_ptr()),
                     C.c_void_p(V.data_ptr()), C.c_void_p(sig.data_ptr()), C.c_void_p(ws.data_ptr()), nbytes.value, s,
                     C.byref(info))
    torch.cuda.synchronize()
    assert rc == 0
    return info.status


@pytest.mark.parametrize("precision,n,n3", [("fp64", 384, 16), ("fp32", 512, 64)])  # sizes at which such products are taken
def test_products_that_give_up(lib, precision, n, n3):
    assert _status(lib, precision, 0, n, n3) == 0
    assert _status(lib, precision, EXPIRE, n, n3) == -3  # TSVD_ERR_CUDA
    assert _status(lib, precision, 0, n, n3) == 0


@pytest.mark.parametrize("precision,n,n3", [("fp64", 384, 16), ("fp32", 512, 64)])
def test_simt_takes_no_such_product(lib, precision, n, n3):
    """TSVD_FLAG_SIMT: no tensor-core product that could give up."""
    assert _status(lib, precision, SIMT | EXPIRE, n, n3) == 0
