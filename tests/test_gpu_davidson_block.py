"""The Davidson subspace kernels at the block sizes where they take another form: 1, 2, 4, 8 and more
vectors per pass, at most 16 and more new vectors at a time (the triangle of the block's Cholesky factor),
vectors in one slice and in several.  Each pair is compared with the dense spin-adapted matrix (columns
of sigma): a residual of S-norm r puts the energy within r of an eigenvalue, and the vectors are
S-orthonormal up to rounding (about 1e-15 per element of the basis, at most some hundreds of them)."""
import numpy as np
import pytest
import scipy.linalg

from adc_inputs import make_system
from oracle.spinadapted import SpinAdaptedADC

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,o,v,naux,nroots", [("ea", 2, 5, 12, 1), ("ip", 4, 7, 20, 2), ("ea", 3, 9, 24, 3), ("ea", 4, 17, 40, 5),
                                                  ("ip", 4, 7, 20, 9), ("ea", 4, 17, 40, 17)])
def test_davidson_blocks_vs_dense(kind, o, v, naux, nroots):
    from paper_2012_06714_gb300 import ADC

    s = make_system(o, v, naux, seed=nroots)
    ref = SpinAdaptedADC(s.eps, o, s.B, 2, kind)
    g = ADC(s.eps, s.B, o, order=2, kind=kind, max_iter=300, res_tol=1e-7)
    S = ref.apply_S(np.eye(g.dim))
    A = g.sigma(np.eye(g.dim)) @ S  # rows: sigma(e_k) S
    w = scipy.linalg.eigh(0.5 * (A + A.T), S, eigvals_only=True)
    e, _, x, st = g.davidson(nroots, tol=1e-10, want_vectors=True)
    assert st["status"] in (0, -4)  # -4: the basis cannot grow any more (9 IP roots), with the residuals below
    assert np.abs(w[None, :] - e[:, None]).min(axis=1).max() <= 1e-7
    assert np.abs(x @ S @ x.T - np.eye(nroots)).max() <= 1e-11
    r = g.sigma(x) - e[:, None] * x
    assert np.sqrt(np.einsum("rx,rx->r", r @ S, r)).max() <= 1.01e-7
    g.close()
