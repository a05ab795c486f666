"""Krylov workspace and kernel limits on the CPU, the CUDA runtime a host stand-in:
after a failed allocation or memset the next solve starts from a complete
workspace (the Gram-Schmidt kernels count their finished blocks in a zeroed word),
and a kernel's shared-memory limit, which all threads of a process share, never
depends on the length of one solve's basis."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CHILD = r"""
import ctypes
import numpy as np
import synth
from tests.helpers import create
from paper_2608_27863_gb300 import hdg as H
fake = ctypes.CDLL(None)
for f in (fake.fake_fail_malloc, fake.fake_fail_memset, fake.fake_cleared):
    f.argtypes = [ctypes.c_size_t]
fake.fake_fill.argtypes = [ctypes.c_double]
L = H.lib()
ptr = lambda a: ctypes.c_void_p(a.ctypes.data)

class Solver:
    def __init__(self, n):
        P = synth.config1(n=n, p=1)
        self.h = create(P)
        self.a = [np.ascontiguousarray(x) for x in (P.U, P.Q, P.UH, P.Ustar)]
        assert L.hdg_linearize_condense(self.h, *map(ptr, self.a), None, P.dt, P.a_ii, None) == H.HDG_OK
        self.b, self.x = np.zeros_like(P.UH), np.zeros_like(P.UH)

    def gmres(self, m):
        it, rel = ctypes.c_int(0), ctypes.c_double(0.0)
        rc = L.hdg_gmres(self.h, ptr(self.b), ptr(self.x), m, m, 1e-300, 0, ctypes.byref(it), ctypes.byref(rel))
        return rc, it.value
"""
FAILURE = CHILD + r"""
s = Solver(3)
before = fake.fake_cleared(4)
fake.fake_fail_%s(4)
assert s.gmres(10)[0] != H.HDG_OK
assert s.gmres(10)[0] == H.HDG_OK
assert fake.fake_cleared(4) == before + 1, "no cleared counter"
L.hdg_destroy(s.h)
print("complete")
"""
LIMITS = CHILD + r"""
fake.fake_fill(1.0)
for m in (500, 330):
    s = Solver(50)
    assert s.b.size > 2 * 152 * 128                  # the wide kernels
    assert s.gmres(m) == (H.HDG_ENOCONV, m)
    L.hdg_destroy(s.h)
assert fake.fake_refused() == 0 and fake.fake_varied() == 0, (fake.fake_refused(), fake.fake_varied())
print("complete")
"""


def run_child(tmp_path, code):
    from paper_2608_27863_gb300 import build
    build.build()
    so = str(tmp_path / "libfake.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", so, os.path.join(HERE, "cuda", "fake_cudart.c")], check=True)
    r = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(HERE), capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=so, PYTHONPATH=os.path.dirname(HERE)))
    assert r.returncode == 0 and "complete" in r.stdout, r.stdout + r.stderr


@pytest.mark.parametrize("what", ["malloc", "memset"])
def test_workspace_is_complete_after_a_failure(tmp_path, what):
    run_child(tmp_path, FAILURE % what)


def test_shared_memory_limits_do_not_depend_on_the_basis(tmp_path):
    run_child(tmp_path, LIMITS)
