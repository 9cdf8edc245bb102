"""FP64 contractions on the tensor cores (exact digit products) against the oracle, through FP64
sigmas: contraction lengths below, at and between multiples of the 32-deep K block and the 128-deep
epoch, tiles of 16 to 64 columns, few and many rows, K slices.  Tolerance: the library's FP64 bound is
1e-11 of max |sigma|; the digit products' error is that of FP64 rounding, so 1e-13 is asked here
(sigma sums some 20 contractions of relative error below 1e-15 each, with cancellation of at most one
order between them)."""
import numpy as np
import pytest

from adc_inputs import make_system
from oracle.spinadapted import SpinAdaptedADC

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,o,v,naux,nvec", [("ea", 2, 17, 33, 1), ("ip", 3, 40, 129, 2), ("ip", 9, 31, 64, 3),
                                                ("ea", 5, 65, 200, 2), ("ip", 17, 20, 128, 9), ("ea", 8, 32, 96, 17)])
@pytest.mark.parametrize("graded", [False, True])
def test_fp64_sigma_on_tensor_cores(kind, o, v, naux, nvec, graded):
    from paper_2012_06714_gb300 import ADC

    s = make_system(o, v, naux, seed=o)
    ref = SpinAdaptedADC(s.eps, o, s.B, 3, kind)
    g = ADC(s.eps, s.B, o, order=3, kind=kind, precision="fp64")
    rng = np.random.default_rng(v)
    X = rng.standard_normal((nvec, g.dim))
    if graded:  # elements over twelve orders of magnitude, one vector all zero
        X *= 10.0 ** rng.uniform(-12.0, 0.0, size=X.shape)
        X[0] = 0.0
    S, R = g.sigma(X), ref.sigma(X)
    g.close()
    assert np.abs(S - R).max() <= 1e-13 * max(np.abs(R).max(), 1e-300)
    if graded:
        assert not S[0].any()


def test_non_finite_rows_stay_apart():
    """A NaN or an infinity in one vector makes that vector's result non-finite and no other's."""
    from paper_2012_06714_gb300 import ADC

    o, v, naux = 6, 40, 120
    s = make_system(o, v, naux, seed=3)
    g = ADC(s.eps, s.B, o, order=3, kind="ea", precision="fp64")
    X = np.random.default_rng(1).standard_normal((3, g.dim))
    R = g.sigma(X)
    X[0, v + 5] = np.nan
    X[2, v + 7] = np.inf
    S = g.sigma(X)
    g.close()
    assert not np.isfinite(S[0, :v]).any() and not np.isfinite(S[2, :v]).any()
    assert np.array_equal(S[1], R[1])


@pytest.mark.parametrize("o,v,nvec", [(2, 16, 260), (3, 14, 260), (4, 16, 130), (2, 23, 90), (4, 32, 20), (2, 46, 17)])
def test_rows_of_a_cluster(o, v, nvec):
    """Contractions of o v^2 = 512, 588, 1024, 1058, 4096 and 4232 terms (ADC(2): the singles row), the
    lengths between which rows are cut into digits by one block, by clusters of up to eight, and in two
    passes.  The bound of the test above."""
    from paper_2012_06714_gb300 import ADC

    s = make_system(o, v, 60, seed=v)
    ref = SpinAdaptedADC(s.eps, o, s.B, 2, "ea")
    g = ADC(s.eps, s.B, o, order=2, kind="ea", precision="fp64")
    X = np.random.default_rng(v).standard_normal((nvec, g.dim))
    S, R = g.sigma(X), ref.sigma(X)
    g.close()
    assert np.abs(S - R).max() <= 1e-13 * np.abs(R).max()


@pytest.mark.parametrize("p", [-1035, -1000, 960])
def test_range_of_doubles(p):
    """Vectors scaled by 2^p, subnormal at -1035: sigma is linear, so it scales with them, to the FP64 bound of
    the tests above and, where results or intermediates are subnormal, a unit 2^-1074 for each of the up to 1e5
    terms that a result sums over all its contractions."""
    from paper_2012_06714_gb300 import ADC

    o, v = 6, 40
    s = make_system(o, v, 120, seed=3)
    g = ADC(s.eps, s.B, o, order=3, kind="ip", precision="fp64")
    X = np.ldexp(np.random.default_rng(5).standard_normal((64, g.dim)), p)
    S, R = g.sigma(X), g.sigma(np.ldexp(X, -p))
    g.close()
    assert np.abs(np.ldexp(S, -p) - R).max() <= 1e-13 * np.abs(R).max() + 1e5 * np.ldexp(1.0, -1074 - p)


@pytest.mark.parametrize("o,v,naux,nvec", [(8, 64, 100, 3), (9, 57, 100, 3), (16, 64, 60, 3), (25, 41, 60, 3), (32, 128, 30, 2), (17, 241, 20, 2)])
def test_digits_of_long_rows(o, v, naux, nvec):
    """Rows of o v = 512, 513, 1024, 1025, 4096 and 4097 terms, between which they are cut into digits by one block,
    by clusters of up to eight, and in two passes: the product Qjc,njcd->nQd of an ADC(2) sigma without the held
    coupling block, of more than the 4e6 flop from which digits are made.  The bound of the tests above."""
    from paper_2012_06714_gb300 import ADC, release_memory

    assert 2 * naux * nvec * v * o * v >= 4e6
    s = make_system(o, v, naux, seed=v)
    ref = SpinAdaptedADC(s.eps, o, s.B, 2, "ea")
    g = ADC(s.eps, s.B, o, order=2, kind="ea", precision="fp64")
    release_memory()  # the coupling block
    X = np.random.default_rng(v).standard_normal((nvec, g.dim))
    S, R = g.sigma(X), ref.sigma(X)
    g.close()
    assert np.abs(S[:, :v] - R[:, :v]).max() <= 1e-13 * np.abs(R[:, :v]).max()
    assert np.abs(S - R).max() <= 1e-13 * np.abs(R).max()
