"""The least workspaces of the products (TSVD_WS_LEAST): what the calls took before their products had
tensor-core forms, by formula; no GPU needed."""
import ctypes as C

import pytest

WS_LEAST = 256


@pytest.fixture(scope="module")
def lib():
    from paper_2504_04989_gb300 import build, _lib
    build.build()
    return _lib.load()


def _size(fn, *args):
    n = C.c_size_t()
    assert fn(*args, C.byref(n)) == 0, args
    return n.value


def _sum(arrays, es):
    return sum((n * es + 255) // 256 * 256 for n in arrays)


@pytest.mark.parametrize("precision,es", [(0, 16), (1, 8)])
@pytest.mark.parametrize("n1,n2,n4,n3", [(64, 48, 32, 16), (1024, 1024, 1024, 64), (45000, 45000, 45000, 1), (3, 5, 7, 9)])
def test_products(lib, precision, es, n1, n2, n4, n3):
    h, sk = n3 // 2 + 1, 1 << 22
    a, b, c = h * n1 * n2, h * n2 * n4, h * n1 * n4
    least = _sum([a, b, c, sk], es)
    assert _size(lib.tprod_workspace_size, n1, n2, n4, n3, precision | WS_LEAST) == least
    assert _size(lib.tprod_workspace_size, n1, n2, n4, n3, precision) >= least
    assert _size(lib.tprod_backward_workspace_size, n1, n2, n4, n3, precision | WS_LEAST) == _sum([a, b, c, a, b, sk], es)


@pytest.mark.parametrize("precision,es", [(0, 16), (1, 8)])
def test_others(lib, precision, es):
    from paper_2504_04989_gb300 import _lib
    n1, n2, n3, R, h = 2000, 1500, 64, 50, 33
    least = _sum([h * n1 * R, h * n2 * R, h * R, h * n1 * n2, 1 << 20], es)
    assert _size(lib.tsvd_lowrank_workspace_size, n1, n2, n3, R, precision | WS_LEAST) == least
    for fn in (lib.tqr_workspace_size, lib.tpinv_workspace_size):
        assert _size(fn, n1, n2, n3, precision | WS_LEAST) <= _size(fn, n1, n2, n3, precision)
    p = _lib.TsvdParams(R=R, P=10, q=2, precision=precision, seed=0, flags=0)
    q = _lib.TsvdParams(R=R, P=10, q=2, precision=precision, seed=0, flags=WS_LEAST)
    assert _size(lib.tsvd_rbk_workspace_size, n1, n2, n3, C.byref(q)) <= _size(lib.tsvd_rbk_workspace_size, n1, n2, n3, C.byref(p))
