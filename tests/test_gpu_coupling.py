"""The held coupling block (the product of sigma's singles row and doubles block with the singles) against
the oracle where its form changes: an FP32 block (more than 2^24 values) with rows that do and do not start
on 16-byte boundaries and with more than eight vectors, and an IP block formed in several slices of the
virtual index (o v^3 > 2^28).  Tolerances: the split-BF16 bound of sigma, 3e-5 of max |sigma|
(test_gpu_mixed.py); FP64 1e-11 of max |sigma|."""
import numpy as np
import pytest

from adc_inputs import make_system
from oracle.spinadapted import SpinAdaptedADC

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,precision,o,v,naux,nvec,tol", [("ea", "bf16x3", 5, 151, 120, 9, 3e-5), ("ea", "bf16x3", 5, 152, 120, 3, 3e-5),
                                                              ("ip", "fp64", 2, 513, 24, 1, 1e-11)])
def test_coupling_block_vs_oracle(kind, precision, o, v, naux, nvec, tol):
    from paper_2012_06714_gb300 import ADC

    s = make_system(o, v, naux, seed=v)
    ref = SpinAdaptedADC(s.eps, o, s.B, 3, kind)
    g = ADC(s.eps, s.B, o, order=3, kind=kind, precision=precision)
    n1 = v if kind == "ea" else o
    X = np.random.default_rng(v).standard_normal((nvec, g.dim))
    X[:, n1:] /= np.sqrt(v)  # singles and doubles parts of sigma of the same order
    S, R = g.sigma(X), ref.sigma(X)
    g.close()
    for part in (slice(0, n1), slice(n1, None)):
        assert np.abs(S[:, part] - R[:, part]).max() <= tol * np.abs(R).max()


@pytest.mark.parametrize("precision,tol", [("bf16x3", 3e-5), ("fp64", 1e-11)])
def test_ea_coupling_block_in_slices_vs_oracle(precision, tol):
    """An EA block formed in two slices of the virtual index, 445 and 3 of 448 (o v^3 > 2^28)."""
    from paper_2012_06714_gb300 import ADC

    o, v = 3, 448
    assert o * v**3 > 2**28
    s = make_system(o, v, 24, seed=v)
    ref = SpinAdaptedADC(s.eps, o, s.B, 3, "ea")
    g = ADC(s.eps, s.B, o, order=3, kind="ea", precision=precision)
    X = np.random.default_rng(v).standard_normal((2, g.dim))
    X[:, v:] /= np.sqrt(v)
    S, R = g.sigma(X), ref.sigma(X)
    g.close()
    for part in (slice(0, v), slice(v, None)):
        assert np.abs(S[:, part] - R[:, part]).max() <= tol * np.abs(R).max()
