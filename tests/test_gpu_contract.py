"""The quad / hex contraction kernel at every instantiated (dim, p), with all of
its terms at once: artificial viscosity (the density row then has a viscous
part), state-dependent tau and boundary faces of several kinds, over element
counts whose last tiles are not full.

FP64: the oracle's blocks within 1e-11, the bar of every parity test.  FP32: the
Schur product's sums of n_u terms err by at most n_u 2^-24 of the terms' size,
of random sign by its root; a block across the element is down to a fortieth of
its terms, the largest block of its row.  4 n_u 2^-24 of every block's own size
(3.8e-6 to 7.6e-5; half precision in the contraction would give 5e-4 and more)."""
import numpy as np
import pytest

import synth
from tests.helpers import GpuRun
from tests.test_gpu_mixed import blocks_of
from tests.test_gpu_parity import compare, tagged

pytestmark = pytest.mark.gpu


def problem(dim, p):
    P = tagged(synth.tiny(dim, p, seed=3, periodic=(False, True, True)[:dim], visc_law=1, av=2e-3),
               {(0, 0): 3, (0, 1): 2}, twall=0.9)
    P.tau_mode = 1
    return P


@pytest.mark.parametrize("dim,p", [(2, 1), (2, 2), (2, 3), (3, 1), (3, 2), (3, 3)])
def test_contraction_matches_oracle_and_mixed_follows(dim, p):
    pytest.importorskip("torch")
    from paper_2608_27863_gb300 import hdg as H
    P = problem(dim, p)
    compare(P, rows=[0, 11, 29, 50] if dim == 3 else None, check_matvec=False)
    run = GpuRun(P)
    run.linearize()
    ref = blocks_of(run, False)
    H.hdg_set_params(run.h, tau=P.tau, visc_law=P.visc_law, suth_c1=P.suth_c1, suth_s=P.suth_s,
                     precision=H.HDG_PREC_MIXED, tau_mode=1)
    run.linearize()
    assert H.hdg_status(run.h) == 0
    mix = blocks_of(run, True)
    run.close()
    errs = np.linalg.norm(mix - ref, axis=(1, 2)) / np.linalg.norm(ref, axis=(1, 2))
    assert errs.max() < 4 * (dim + 2) * (p + 1) ** dim * 2.0 ** -24, errs.max()
