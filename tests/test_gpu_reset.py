"""Products before and after the device's context is reset, in a process of its
own: what the library keeps between calls (the scratch pool, kernel
attributes, addresses) must not outlive the context."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU machine
    pytest.skip("no GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes
import numpy as np
import bitgen, oracle as O
import paper_1909_01554_gb300 as bmm

L = bmm.lib()
runtime = ctypes.CDLL(None)
if not hasattr(runtime, "cudaMalloc"):  # libbmm's own copy, by the name it was loaded under
    with open("/proc/self/maps") as f:
        path = next(l.split()[-1] for l in f if "libcudart" in l)
    runtime = ctypes.CDLL(path)

def check(e):
    assert e == 0, e

def device(words):
    p = ctypes.c_void_p()
    check(runtime.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(words.nbytes)))
    check(runtime.cudaMemcpy(p, words.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(words.nbytes), 1))
    return p

def products(seed):
    m, k, n = 1152, 1664, 1280  # leaves of one level: k padded
    A, B = bitgen.fill_cpu(m, k, seed, 0), bitgen.fill_cpu(k, n, seed, 1)
    want = O.cubic(O.GF2, A, B, m, k, n)
    a, b = device(A), device(B)
    def run(f):
        C = np.zeros((m, n // 64), dtype=np.uint64)
        c = device(C)
        check(f(c))
        check(L.bmm_stream_status(None))
        check(runtime.cudaMemcpy(C.ctypes.data_as(ctypes.c_void_p), c, ctypes.c_size_t(C.nbytes), 2))
        assert (C == want).all()
    for o in (bmm.opts(), bmm.opts(path=bmm.PATH_POPC, depth=0), bmm.opts(path=bmm.PATH_TC_FP4_PAIR, depth=0),
              bmm.opts(depth=1), bmm.opts(depth=1, serial=1)):
        run(lambda c: L.bmm_gf2_ex(a, b, c, m, k, n, ctypes.byref(o), None))
    run(lambda c: L.bmm_product_noalloc(0, a, b, c, m, k, n, None))

products(1)
L.bmm_host_release()
check(runtime.cudaDeviceReset())
products(2)
check(runtime.cudaDeviceReset())
products(3)
print("done")
"""


def test_products_after_a_device_reset():
    import paper_1909_01554_gb300 as bmm

    if not bmm.device_supported():
        pytest.skip("tensor-core paths need sm_103")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env={**os.environ, "PYTHONPATH": os.pathsep.join([ROOT])},
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stderr[-2000:]
