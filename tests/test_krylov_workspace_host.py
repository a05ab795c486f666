"""The Krylov workspace after a failed allocation or memset, on the CPU with a
host stand-in for the CUDA runtime: the next solve starts from a complete
workspace (the Gram-Schmidt kernels count their finished blocks in a zeroed word)."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CHILD = r"""
import ctypes, sys
import numpy as np
import synth
from tests.helpers import create
from paper_2608_27863_gb300 import hdg as H
fake = ctypes.CDLL(None)
for f in (fake.fake_fail_malloc, fake.fake_fail_memset, fake.fake_cleared):
    f.argtypes = [ctypes.c_size_t]
P = synth.config1(n=3, p=1)
h = create(P)
ptr = lambda a: ctypes.c_void_p(a.ctypes.data)
a = [np.ascontiguousarray(x) for x in (P.U, P.Q, P.UH, P.Ustar)]
L = H.lib()
assert L.hdg_linearize_condense(h, *map(ptr, a), None, P.dt, P.a_ii, None) == H.HDG_OK
b, x = np.zeros_like(a[2]), np.zeros_like(a[2])
it, rel = ctypes.c_int(0), ctypes.c_double(0.0)
gmres = lambda: L.hdg_gmres(h, ptr(b), ptr(x), 10, 10, 1e-8, 0, ctypes.byref(it), ctypes.byref(rel))
before = fake.fake_cleared(4)
getattr(fake, "fake_fail_" + sys.argv[1])(4)
assert gmres() != H.HDG_OK
assert gmres() == H.HDG_OK
assert fake.fake_cleared(4) == before + 1, "no cleared counter"
L.hdg_destroy(h)
print("complete")
"""


@pytest.mark.parametrize("what", ["malloc", "memset"])
def test_workspace_is_complete_after_a_failure(tmp_path, what):
    from paper_2608_27863_gb300 import build
    build.build()
    so = str(tmp_path / "libfake.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", so, os.path.join(HERE, "cuda", "fake_cudart.c")], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD, what], cwd=os.path.dirname(HERE), capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=so, PYTHONPATH=os.path.dirname(HERE)))
    assert r.returncode == 0 and "complete" in r.stdout, r.stdout + r.stderr
