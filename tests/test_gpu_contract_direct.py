"""The contraction kernel on one element with coefficients given here, its FP32
instance against the FP64 one and against sums that the mixed form holds in FP64."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def contract(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_27863_gb300 import build as b
    so = str(tmp_path_factory.mktemp("contract") / "libcontract.so")
    r = subprocess.run([b._nvcc()] + b.ARCH + b.FLAGS + ["-I" + b.CSRC, "-shared", "-o", so,
                        os.path.join(HERE, "cuda", "contract_direct.cu"), "-x", "cu", os.path.join(b.CSRC, "refelem.cpp"),
                        "-lcudart"], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    fn = ctypes.CDLL(so).contract_one

    def call(d, p, fp32, vcoef, fcoef, taup, dt, tau):
        m, nf = d + 2, 2 * d
        nu, nt = m * (p + 1) ** d, nf * m * (p + 1) ** (d - 1)
        # a cell of unequal sides: det J, d xi_r / d x_k, outward area vectors per reference face
        h = np.array([0.5, 0.3, 0.8])[:d] / 2
        det = h.prod()
        nw = np.zeros((nf, d))
        for f in range(nf):
            nw[f, f // 2] = (1 if f & 1 else -1) * det / h[f // 2]
        geo = np.concatenate([[det], np.diag(1 / h).ravel(), nw.ravel()])
        out = [np.zeros(s) for s in ((nu, nu), (nu, nt), (nt, nu), (nt, nt))]
        arrs = [np.ascontiguousarray(a, dtype=np.float64) for a in (vcoef, fcoef, taup, geo)]
        ptr = lambda a: ctypes.c_void_p(a.ctypes.data)
        rc = fn(d, p, int(fp32), *[ptr(a) for a in arrs], ctypes.c_double(dt), ctypes.c_double(np.inf),
                ctypes.c_double(tau), *[ptr(a) for a in out])
        assert rc == 0
        return out

    return call


def coefficients(d, p, seed):
    m, nf, nq, nfq = d + 2, 2 * d, (p + 2) ** d, (p + 2) ** (d - 1)
    rng = np.random.default_rng(seed)
    vol = rng.normal(size=(m * m, d, 1 + d, nq)).astype(np.float32).astype(float)
    face = rng.normal(size=(nf, m * m, 1 + d, nfq)).astype(np.float32).astype(float)
    return vol, face, rng.uniform(1, 5, size=(nf, nfq))


@pytest.mark.parametrize("d", [2, 3])
def test_interior_block_adds_volume_and_face_parts_in_fp64(contract, d):
    """a_ii = inf (no mass term): the block of both parts is the sum of the parts' blocks, each an FP32 sum, to FP64
    rounding; a sum of the two in FP32 misses by 2^-24 of it."""
    p, dt = 2, 0.37
    vol, face, tau = coefficients(d, p, d)
    both = contract(d, p, True, vol, face, tau, dt, 0.0)[0]
    v = contract(d, p, True, vol, 0 * face, 0 * tau, dt, 0.0)[0]
    f = contract(d, p, True, 0 * vol, face, tau, dt, 0.0)[0]
    assert np.abs(f).max() > 0 and np.abs(v).max() > 0
    assert (np.abs(both - (v + f)) <= 2.0 ** -51 * (np.abs(v) + np.abs(f))).all()


@pytest.mark.parametrize("d", [2, 3])
def test_tau_weighted_face_mass_is_rounded_once(contract, d):
    """State-dependent tau: without flux coefficients the trace rows hold |n| sum_s w tau mu mu, summed in FP64 and
    rounded to FP32 once (2^-24); a sum in FP32 has (p + 2)^(d - 1) roundings."""
    vol, face, tau = coefficients(d, 2, d)
    ref = contract(d, 2, False, 0 * vol, 0 * face, tau, 0.37, 0.0)[2]
    got = contract(d, 2, True, 0 * vol, 0 * face, tau, 0.37, 0.0)[2]
    assert np.abs(ref).max() > 0
    assert (np.abs(got - ref) <= (2.0 ** -24 + 1e-14) * np.abs(ref)).all()


@pytest.mark.parametrize("d", [2, 3])
def test_fp32_blocks_follow_fp64_before_elimination(contract, d):
    """All four blocks of the FP32 instance against the FP64 one.  An entry passes through about 20 sums, one axis at a
    time and then dt times the face rows, of terms of random sign: 20^(1/2) 2^-24 = 2.7e-7 of its size, four times
    which is the bar (half precision would miss it by 2^13)."""
    args = coefficients(d, 2, 10 + d) + (0.37, 2.5)
    ref, got = contract(d, 2, False, *args), contract(d, 2, True, *args)
    for a, b in zip(ref, got):
        assert np.linalg.norm(b - a) <= 1.1e-6 * np.linalg.norm(a)
