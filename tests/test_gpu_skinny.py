"""The bandwidth kernels of the few-vector products for every number of vectors they are compiled for (1 to 8),
with rows of the large operand that start on 16-byte boundaries and rows that do not, and sizes that leave part
of a block, of a K slice and of a 64-term partial sum over: the products of sigma with the FP32 coupling block
(more than 2^24 values), against the oracle.  Tolerance: the split-BF16 bound of sigma, 3e-5 of max |sigma|
(test_gpu_mixed.py), for the singles and the doubles part separately."""
import numpy as np
import pytest

from adc_inputs import make_system
from oracle.spinadapted import SpinAdaptedADC

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("o,v,naux", [(5, 153, 40), (5, 154, 40), (4, 168, 40)])
def test_every_number_of_vectors_vs_oracle(o, v, naux):
    from paper_2012_06714_gb300 import ADC

    s = make_system(o, v, naux, seed=v)
    ref = SpinAdaptedADC(s.eps, o, s.B, 3, "ea")
    g = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3")
    X = np.random.default_rng(v).standard_normal((8, g.dim))
    X[:, v:] /= np.sqrt(v)  # singles and doubles parts of sigma of the same order
    R = ref.sigma(X)
    for n in range(1, 9):
        S = g.sigma(X[:n])
        for part in (slice(0, v), slice(v, None)):
            assert np.abs(S[:, part] - R[:n, part]).max() <= 3e-5 * np.abs(R[:n]).max(), n
    g.close()


@pytest.mark.parametrize("o,v,naux", [(5, 216, 40), (5, 217, 40)])
def test_one_and_two_vectors_vs_oracle(o, v, naux):
    """One and two vectors at sizes whose coupling products reach the bandwidth kernels (1e8 flop for one vector;
    at the sizes above they are smaller and taken in FP64)."""
    from paper_2012_06714_gb300 import ADC

    s = make_system(o, v, naux, seed=v)
    ref = SpinAdaptedADC(s.eps, o, s.B, 3, "ea")
    g = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3")
    X = np.random.default_rng(v).standard_normal((2, g.dim))
    X[:, v:] /= np.sqrt(v)
    R = ref.sigma(X)
    for n in (1, 2):
        assert 2.0 * n * o * v**3 >= 1e8
        S = g.sigma(X[:n])
        for part in (slice(0, v), slice(v, None)):
            assert np.abs(S[:, part] - R[:n, part]).max() <= 3e-5 * np.abs(R[:n]).max(), n
    g.close()
