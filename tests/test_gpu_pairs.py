"""The ladder over pair-adapted integrals (sigma and setup of mixed-precision handles) against the
oracle at the sizes where its index arithmetic can go wrong: pair counts that are and are not
multiples of the 8-element row padding (P = v (v + 1) / 2), of the 32 x 32 packing and 16 x 16
unfolding tiles and of the 256-row GEMM tile, one and several matrices.  Tolerance: the split-BF16
bound of sigma, 3e-5 of max |sigma| (test_gpu_mixed.py); t2(2), three planes, 1e-6 of its maximum."""
import numpy as np
import pytest

from adc_inputs import make_system
from oracle.spinadapted import SpinAdaptedADC

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("o,v,naux,nvec", [(2, 1, 5, 1), (2, 2, 7, 3), (2, 15, 40, 1), (3, 16, 60, 2), (4, 31, 90, 1),
                                           (4, 33, 100, 3), (5, 48, 130, 2), (4, 65, 200, 4)])
def test_pair_ladder_vs_oracle(o, v, naux, nvec):
    from paper_2012_06714_gb300 import ADC

    s = make_system(o, v, naux, seed=v)
    ref = SpinAdaptedADC(s.eps, o, s.B, 3, "ea")
    g = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3")
    t2 = g.get("t2_2", (o, o, v, v))
    assert np.abs(t2 - ref.t_2).max() <= 1e-6 * np.abs(ref.t_2).max()
    X = np.random.default_rng(v).standard_normal((nvec, g.dim))
    S, R = g.sigma(X), ref.sigma(X)
    scale = max(np.abs(R).max(), np.abs(ref.ladder(X[:, v:].reshape(nvec, o, v, v))).max())
    assert np.abs(S - R).max() <= 3e-5 * scale
    g.close()


def test_pair_integrals_are_given_back():
    """A handle's pair integrals go back to the device when another handle's allocation fails; its
    sigma then takes the two-GEMM form and stays within the split-BF16 bound."""
    from paper_2012_06714_gb300 import ADC

    o, v, naux = 6, 160, 200
    s = make_system(o, v, naux, seed=1)
    a = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3")
    X = np.random.default_rng(2).standard_normal((4, a.dim))
    before = a.sigma(X)
    pairs = 8 * (v * (v + 1) // 2) ** 2  # two planes of both halves
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (900 << 20), dtype=torch.uint8, device="cuda")
    try:
        b = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3")  # needs more than the 900 MB left
        left, _ = torch.cuda.mem_get_info()
        assert left < (900 << 20) + pairs
        Sb = b.sigma(X)
        after = a.sigma(X)
        b.close()
    finally:
        del hold
        torch.cuda.empty_cache()
    tol = 3e-5 * np.abs(before).max()
    assert np.abs(after - before).max() <= tol and np.abs(Sb - before).max() <= tol
    a.close()


def test_out_of_memory_leaves_the_handle_usable():
    """A block of vectors too large for the device is refused with ADC_ERR_OOM after the handle gave back what
    it held for speed, and later calls are right (sigma's split-BF16 bound)."""
    from paper_2012_06714_gb300 import ADC
    from paper_2012_06714_gb300._lib import ADCError

    o, v, naux = 6, 160, 200
    s = make_system(o, v, naux, seed=1)
    a = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3")
    X = np.random.default_rng(2).standard_normal((400, a.dim))  # 0.49 GB, and more than four times that as scratch
    before = a.sigma(X[:4])
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (200 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(ADCError) as e:
            a.sigma(X)
        assert e.value.code == -2
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.abs(a.sigma(X[:4]) - before).max() <= 3e-5 * np.abs(before).max()
    a.close()


@pytest.mark.parametrize("precision,nvec,tol", [("bf16x3", 826, 3e-5), ("fp64", 331, 1e-11)])
def test_matrices_in_groups(precision, nvec, tol):
    """More matrices than one group of the pair ladder takes (at 180 virtuals 8240 in mixed precision and 3295 in
    FP64): the first, the middle and the last vectors of the block against the same vectors by themselves."""
    from paper_2012_06714_gb300 import ADC

    o, v, naux = 10, 180, 300
    s = make_system(o, v, naux, seed=1)
    g = ADC(s.eps, s.B, o, order=3, kind="ea", precision=precision)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(7)
    X = torch.randn(nvec, g.dim, dtype=torch.float64, device="cuda", generator=gen)
    S = g.sigma(X)
    pick = [0, 1, nvec // 2, nvec - 3, nvec - 2, nvec - 1]
    R = g.sigma(X[pick].contiguous())
    assert float((S[pick] - R).abs().max()) <= tol * float(R.abs().max())
    g.close()
