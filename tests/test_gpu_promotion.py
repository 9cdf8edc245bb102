"""Products of few tiles promote their FP32 partial sums often enough.  The tensor core's accumulator truncates,
by about a quarter of its last place per MMA, so sums that run too long shift sigma toward zero.  At 13 / 97 /
385 with six vectors the ring products have 5 tiles of 20 K blocks.  Summed two blocks at a time, 24 MMAs of
which 8 are at full size, the shift is at most 8 * 2^-24 / 4 = 1.2e-7 of a partial sum, and on average over
sums of random sign below a tenth of that; eight blocks at a time it is 2.5e-8.  Asked: a relative bias of at
most 1.2e-8, and an error no larger than the 2.744e-7 that the same sigma had when every such product was cut
into K slices of two blocks (2% for the order of the sums)."""
import numpy as np
import pytest

from adc_inputs import make_system
from oracle.spinadapted import SpinAdaptedADC

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_products_of_few_tiles_are_not_biased():
    from paper_2012_06714_gb300 import ADC

    o, v, naux, n = 13, 97, 385, 6
    s = make_system(o, v, naux, seed=7)
    ref = SpinAdaptedADC(s.eps, o, s.B, 3, "ip")
    g = ADC(s.eps, s.B, o, order=3, kind="ip", precision="bf16x3")
    X = np.random.default_rng(7).standard_normal((n, g.dim)) / np.sqrt(g.dim)
    R = ref.sigma(X)
    d = g.sigma(X) - R
    g.close()
    assert abs((d * R).sum()) <= 1.2e-8 * (R * R).sum()
    assert np.linalg.norm(d) <= 1.02 * 2.744e-7 * np.linalg.norm(R)
