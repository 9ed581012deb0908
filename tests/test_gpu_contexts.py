"""A context that is destroyed and made again: kernels that use more than 48 KB of shared memory are allowed to in each.
In a process of its own, without torch's context."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
import ctypes, sys
import numpy as np
from paper_2607_17419_b200 import binding as kb
cu = ctypes.CDLL("libcuda.so.1")
def ok(r):
    assert r == 0, r
u64, byref = ctypes.c_uint64, ctypes.byref
ok(cu.cuInit(0))
T, d = 512, 16
rng = np.random.default_rng(0)
host = [rng.standard_normal((1, 2, T, d)).astype(np.float32) for _ in range(3)]
results = []
for _ in range(2):
    ctx = ctypes.c_void_p()
    ok(cu.cuCtxCreate_v2(byref(ctx), 0, 0))
    ptrs = []
    for a in host + [np.zeros_like(host[0])]:
        p = u64()
        ok(cu.cuMemAlloc_v2(byref(p), ctypes.c_size_t(a.nbytes)))
        ok(cu.cuMemcpyHtoD_v2(p, a.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(a.nbytes)))
        ptrs.append(p)
    o = kb.make_opts(kb.KATA_F32)
    st = kb.lib().kata_fwd_chunked(*(p.value for p in ptrs), 1, 2, T, d, d, 64, byref(o))
    ok(cu.cuCtxSynchronize())
    out = np.empty_like(host[0])
    ok(cu.cuMemcpyDtoH_v2(out.ctypes.data_as(ctypes.c_void_p), ptrs[3], ctypes.c_size_t(out.nbytes)))
    results.append((st, out))
    ok(cu.cuCtxDestroy_v2(ctx))
assert [st for st, _ in results] == [0, 0], [st for st, _ in results]
assert np.abs(results[0][1]).max() > 0 and np.array_equal(results[0][1], results[1][1])
print("both contexts ran")
"""


def test_a_second_context():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, env=dict(os.environ, PYTHONPATH=root), capture_output=True, text=True,
                       timeout=240)
    assert r.returncode == 0 and "both contexts ran" in r.stdout, r.stdout + r.stderr
