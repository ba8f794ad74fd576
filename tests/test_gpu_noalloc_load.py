"""tprod_noalloc loads all it can need at its first call: calls of other lengths, sizes
and precisions take no device memory afterwards (lazy loading, a process of its own)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import ctypes as C
import torch
from paper_2504_04989_gb300 import _lib
lib = _lib.load()
buf = {c: [torch.randn(1 << 20, device="cuda").to(t) for _ in range(3)] for c, t in ((0, torch.float64), (1, torch.float32))}
torch.cuda.synchronize()
def call(n1, n2, n4, n3, code):
    a, b, c = (C.c_void_p(x.data_ptr()) for x in buf[code])
    assert lib.tprod_noalloc(a, b, c, n1, n2, n4, n3, code, C.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
call(8, 8, 8, 16, 1)
before = torch.cuda.mem_get_info()[0]
for code in (1, 0):
    for n3 in (1, 2, 4, 8, 32, 64, 128, 3, 31, 100, 162, 375, 811):
        call(8, 8, 8, n3, code)
    call(200, 300, 200, 3, code)
    call(250, 1024, 40, 2, code)
print("TAKEN", before - torch.cuda.mem_get_info()[0])
"""


def test_one_call_loads_all():
    import __graft_entry__ as g
    g.build()
    env = dict(os.environ, CUDA_MODULE_LOADING="LAZY", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, cwd=ROOT, env=env, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    taken = int(r.stdout.split("TAKEN")[1])
    assert taken <= 0, taken
