"""The mixed form's 3xTF32 Schur product against the FP32 SIMT one, for every
tile shape (dim, p): one to four column tiles, row and K tails, rows whose
padded stride differs from their length (hex p = 2).

Both start from the same FP32 W, Z and D.  The blocks: FP32 sums of K = n_u
products err by at most K 2^-24 of |W||Z|, the tensor cores' by K / 8
truncations of 2^-23 and the dropped low x low product (2^-22), together
(5 K / 8 + 2) 2^-23.  |W||Z| of a block is measured by the largest block of its
row: the small blocks (a face and the one across the element) are differences of
a D and a WZ of that size, down to a fortieth of it.  Against their own size all
blocks keep 4 K 2^-24: roundings of random sign, a root of K of them, times forty.
The right-hand side: FP64 sums of the same K products in another order."""
import numpy as np
import pytest

import synth
from oracle.hdg import Problem
from tests.helpers import GpuRun
from tests.test_gpu_mixed import blocks_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 2), (2, 3), (3, 1), (3, 2), (3, 3)])
def test_tensor_core_schur_product_follows_fp32(dim, p):
    pytest.importorskip("torch")
    from paper_2608_27863_gb300 import hdg as H
    P = synth.tiny(dim, p, seed=5, visc_law=1, av=1e-3)
    run = GpuRun(P)
    H.hdg_set_params(run.h, tau=P.tau, visc_law=P.visc_law, suth_c1=P.suth_c1, suth_s=P.suth_s,
                     precision=H.HDG_PREC_MIXED)
    out = []
    for mode in (0, 2):
        H.hdg_set_tuning(run.h, schur_mode=mode)
        run.linearize()
        assert H.hdg_status(run.h) == 0
        out.append((blocks_of(run, True), run.rhs()))
    run.close()
    (s0, g0), (s2, g2) = out
    rowptr = Problem(P).conn.rowptr
    size = np.maximum.reduceat(np.linalg.norm(s0, axis=(1, 2)), rowptr[:-1])
    diff, K = np.linalg.norm(s2 - s0, axis=(1, 2)), (dim + 2) * (p + 1) ** dim
    errs = diff / np.repeat(size, np.diff(rowptr))
    assert errs.max() < (5 * K / 8 + 2) * 2.0 ** -23, errs.max()
    own = diff / np.linalg.norm(s0, axis=(1, 2))
    assert own.max() < 4 * K * 2.0 ** -24, own.max()
    assert np.linalg.norm(g2 - g0) <= 1e-11 * np.linalg.norm(g0)
