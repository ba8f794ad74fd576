"""Calls with the least workspace (TSVD_WS_LEAST), with sizes between and with less, and the Python
layer where the device has not more left."""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

WS_LEAST = 256


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2504_04989_gb300 import api as a
    return a


def _ptr(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("precision,code,dt,u", [("fp64", 0, torch.float64, 2.0 ** -53), ("fp32", 1, torch.float32, 2.0 ** -24)])
def test_tprod_sizes(api, precision, code, dt, u):
    """The same product from any accepted size, to 16 u in norm (the forms' own errors are below 14 u and 2 u);
    refused below the least."""
    from paper_2504_04989_gb300 import _lib
    lib = _lib.load()
    n1, n2, n4, n3 = 1100, 1200, 1300, 16
    g = torch.Generator(device="cuda").manual_seed(2)
    A = torch.randn((n3, n1, n2), generator=g, device="cuda", dtype=dt)
    B = torch.randn((n3, n2, n4), generator=g, device="cuda", dtype=dt)
    n = C.c_size_t()
    assert lib.tprod_workspace_size(n1, n2, n4, n3, code, C.byref(n)) == 0
    best = n.value
    assert lib.tprod_workspace_size(n1, n2, n4, n3, code | WS_LEAST, C.byref(n)) == 0
    least = n.value
    assert least < best
    s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    want = api.tprod(A, B, precision)
    for size in (least, least + (best - least) // 3, best - 256, best):
        ws = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        ws[size:] = 77  # the bytes behind stay as they are
        out = torch.empty((n3, n1, n4), dtype=dt, device="cuda")
        assert lib.tprod(_ptr(A), _ptr(B), _ptr(out), n1, n2, n4, n3, code, _ptr(ws), size, s) == 0
        assert float((out - want).norm() / want.norm()) <= 16 * u
        assert bool((ws[size:] == 77).all())
    out = torch.empty((n3, n1, n4), dtype=dt, device="cuda")
    assert lib.tprod(_ptr(A), _ptr(B), _ptr(out), n1, n2, n4, n3, code, _ptr(ws), least - 256, s) == -2


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_tsvd_least(api, precision):
    """A T-SVD, one by one and batched, in the least workspace: singular values to 1e-9 / 1e-4 of the largest, as
    accurate as those of two forms of the same products are bound to agree."""
    from paper_2504_04989_gb300 import _lib
    lib = _lib.load()
    n1, n2, n3, R = 300, 280, 24, 20
    dt = torch.float64 if precision == "fp64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn((n3, n1, n2), generator=g, device="cuda", dtype=dt)
    want = api.rbk(A, R, P=10, q=2, precision=precision)[3]
    plan = api.RbkPlan(n1, n2, n3, R, P=10, q=2, precision=precision)
    p = _lib.TsvdParams.from_buffer_copy(plan.p)
    p.flags |= WS_LEAST
    n = C.c_size_t()
    assert lib.tsvd_rbk_workspace_size(n1, n2, n3, C.byref(p), C.byref(n)) == 0
    plan.nbytes = n.value
    plan.ws = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    got = plan(A)[3]
    tol = 1e-9 if precision == "fp64" else 1e-4
    assert float((got - want).abs().max()) <= tol * float(want.max())
    batch = api.RbkBatchPlan([(n1, n2, n3)] * 3, R, P=10, q=2, precision=precision, lanes=2)
    for d in batch.descs:
        d.params.seed = 0
    for d in batch.descs:
        d.params.flags |= WS_LEAST
    assert lib.tsvd_rbk_batched_workspace_size(batch.descs, 3, 2, C.byref(n)) == 0
    for d in batch.descs:
        d.params.flags &= ~WS_LEAST
    batch.nbytes = n.value
    batch.ws = torch.empty(n.value, dtype=torch.uint8, device="cuda")
    for got in batch([A, A, A])[3]:
        assert float((got - want).abs().max()) <= tol * float(want.max())


def test_device_nearly_full(api):
    """Where the full workspace does not fit, the call takes the least one."""
    from paper_2504_04989_gb300 import _lib
    lib = _lib.load()
    n1, n2, n4, n3 = 2048, 2048, 2048, 3
    n = C.c_size_t()
    lib.tprod_workspace_size(n1, n2, n4, n3, 0, C.byref(n))
    best = n.value
    lib.tprod_workspace_size(n1, n2, n4, n3, WS_LEAST, C.byref(n))
    least = n.value
    A = torch.randn((n3, n1, n2), device="cuda", dtype=torch.float64)
    want = api.tprod(A, A, "fp64")
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    held = torch.cuda.memory_reserved()
    torch.cuda.set_per_process_memory_fraction((held + (least + best) / 2 + want.nbytes) / total)
    try:
        got = api.tprod(A, A, "fp64")
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert float((got - want).norm() / want.norm()) <= 16 * 2.0 ** -53
