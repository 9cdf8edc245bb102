"""Every call that can launch a tensor-core contraction reads the flag that its bounded device waits raise when
they give up: the call returns ADC_ERR_TIMEOUT, keeps nothing of what it formed, and the next one is right.
No wait gives up here: the library is told to find the flag raised at the named reading."""
import numpy as np
import pytest

from adc_inputs import make_open_shell_system, make_system
from oracle.spinadapted import SpinAdaptedADC

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TIMEOUT = -5
O, V, NAUX = 5, 30, 90


def _raise_at(where):
    from paper_2012_06714_gb300 import load_library

    load_library().adc_internal_raise_timeout(where.encode())


def _timeout(call):
    from paper_2012_06714_gb300._lib import ADCError

    with pytest.raises(ADCError) as e:
        call()
    assert e.value.code == TIMEOUT


@pytest.mark.parametrize("precision", ["fp64", "bf16x3"])
def test_calls_of_a_handle(precision):
    from paper_2012_06714_gb300 import ADC

    s = make_system(O, V, NAUX, seed=1)
    ref = SpinAdaptedADC(s.eps, O, s.B, 3, "ea")
    X = np.random.default_rng(1).standard_normal((3, V + O * V * V))
    R = ref.sigma(X)
    tol = (1e-11 if precision == "fp64" else 3e-5) * np.abs(R).max()

    def make(**options):
        return ADC(s.eps, s.B, O, order=3, kind="ea", precision=precision, **options)

    _raise_at("adc_setup")
    _timeout(make)
    _raise_at("adc_setup")
    _timeout(lambda: make(m11_on_the_fly=1))
    g = make()
    good = g.davidson(2, tol=1e-9)
    _raise_at("adc_sigma")
    _timeout(lambda: g.sigma(X))
    assert np.abs(g.sigma(X) - R).max() <= tol
    _raise_at("adc_davidson")
    _timeout(lambda: g.davidson(2, tol=1e-9))
    again = g.davidson(2, tol=1e-9)
    assert np.array_equal(again[0], good[0]) and np.array_equal(again[1], good[1])
    _raise_at("adc_mlp_samples")
    _timeout(lambda: g.mlp_samples(1, iters=(2,), per_vector=10))
    t1 = g.get("t1_3", (O, V))  # (kept since the first solve)
    g.close()
    for call, where in (("get", "t1(3)"), ("get", "adc_get_tensor"), ("davidson", "t1(3)")):
        g = make()
        _raise_at(where)
        _timeout((lambda: g.get("t1_3", (O, V))) if call == "get" else (lambda: g.davidson(2, tol=1e-9)))
        assert np.array_equal(g.get("t1_3", (O, V)), t1)
        g.close()


def test_open_shells():
    from paper_2012_06714_gb300 import ADCUnrestricted

    na, nb, nmo = 5, 4, 23
    s = make_open_shell_system(na, nb, nmo, 41, seed=2)

    def make():
        return ADCUnrestricted(s.eps_a, s.eps_b, s.B_a, s.B_b, na, nb, order=3, kind="ip")

    _raise_at("adc_setup_unrestricted")
    _timeout(make)
    g = make()
    _raise_at("t1(3)")
    _timeout(lambda: g.davidson(2, tol=1e-8))
    shape = (na + nb, 2 * nmo - na - nb)
    t1 = g.get("t1_3", shape)
    g.close()
    g = make()
    assert np.array_equal(g.get("t1_3", shape), t1)
    _raise_at("adc_sigma")
    _timeout(lambda: g.sigma(np.ones((1, g.dim))))
    g.close()
