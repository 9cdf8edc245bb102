"""Memory held for speed under an exhausted device: two host threads, one making small FP64 handles and using
their held coupling blocks, the other making a handle whose setup does not fit what is left, so that its
allocations take back whatever no call keeps.  Every result that is returned is right; running out of memory
(ADC_ERR_OOM) is an answer too.  Tolerances: 1e-11 of max |sigma| in FP64, the split-BF16 bound 3e-5
(test_gpu_mixed.py) in mixed precision."""
import threading

import numpy as np
import pytest

from adc_inputs import make_system
from oracle.spinadapted import SpinAdaptedADC

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_two_host_threads_on_an_exhausted_device():
    from paper_2012_06714_gb300 import ADC
    from paper_2012_06714_gb300._lib import ADCError

    small, big = make_system(4, 18, 60, seed=1), make_system(6, 160, 200, seed=1)
    Xs = np.random.default_rng(1).standard_normal((3, 4 + 16 * 18))
    Xb = np.random.default_rng(2).standard_normal((4, 160 + 6 * 160 * 160))
    Rs = SpinAdaptedADC(small.eps, 4, small.B, 3, "ip").sigma(Xs)
    g = ADC(big.eps, big.B, 6, order=3, kind="ea", precision="bf16x3")
    Rb = g.sigma(Xb)
    g.close()
    right, wrong = {"small": 0, "big": 0}, []

    def use(name, rounds, sys, nocc, kind, precision, X, R, tol, sigmas):
        for _ in range(rounds):
            h = None
            try:
                h = ADC(sys.eps, sys.B, nocc, order=3, kind=kind, precision=precision)
                for _ in range(sigmas):
                    d = np.abs(h.sigma(X) - R).max()
                    if d <= tol * np.abs(R).max():
                        right[name] += 1
                    else:
                        wrong.append((name, d))
            except ADCError as e:
                if e.code != -2:
                    wrong.append((name, str(e)))
            finally:
                if h is not None:
                    h.close()

    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (1300 << 20), dtype=torch.uint8, device="cuda")
    try:
        threads = [threading.Thread(target=use, args=("small", 30, small, 4, "ip", "fp64", Xs, Rs, 1e-11, 4)),
                   threading.Thread(target=use, args=("big", 8, big, 6, "ea", "bf16x3", Xb, Rb, 3e-5, 2))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert not wrong, wrong[:3]
    use("small", 1, small, 4, "ip", "fp64", Xs, Rs, 1e-11, 1)
    use("big", 1, big, 6, "ea", "bf16x3", Xb, Rb, 3e-5, 1)
    assert not wrong and right["small"] >= 1 and right["big"] >= 1, (right, wrong)


def test_samples_with_graphs_when_memory_runs_out():
    """adc_mlp_samples solves like adc_davidson: with cuda_graphs the replayed sigmas hold the pair integrals'
    address, which no allocation of the same call may then take back.  The same samples as from plain launches
    (equal kernels, so equal to rounding: 1e-9 of their maximum)."""
    from paper_2012_06714_gb300 import ADC

    o, v = 3, 40
    s = make_system(o, v, 120, seed=5)
    stream = torch.cuda.Stream()
    got = []
    for graphs in (0, 1):
        g = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3", cuda_graphs=graphs)
        g.set_stream(stream.cuda_stream)
        free, _ = torch.cuda.mem_get_info()
        hold = torch.empty(free - (600 << 20), dtype=torch.uint8, device="cuda")
        try:
            got.append(g.mlp_samples(2, iters=(2, 4), per_vector=500, seed=3))
        finally:
            del hold
            torch.cuda.empty_cache()
        g.close()
    for a, b in zip(*got):
        assert np.abs(a.astype(float) - b).max() <= 1e-9 * max(np.abs(a).max(), 1e-300)


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_the_last_handle_gives_everything_back():
    """adc_destroy releases all of a handle's device memory: with no handle left the device has as much free
    memory as before the handle was made (8 MB for what the driver itself keeps)."""
    from paper_2012_06714_gb300 import ADC, release_memory

    s = make_system(6, 160, 200, seed=1)

    def use():
        g = ADC(s.eps, s.B, 6, order=3, kind="ea", precision="bf16x3")
        g.sigma(np.ones((2, g.dim)))
        g.close()

    use()  # (loads the kernels)
    release_memory()
    free = _free()
    use()
    assert _free() >= free - (8 << 20)


def test_release_memory():
    """adc_release_memory gives back what an idle handle holds for speed, and sigma goes on without it within the
    split-BF16 bound."""
    from paper_2012_06714_gb300 import ADC, release_memory

    o, v = 6, 160
    s = make_system(o, v, 200, seed=1)
    g = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3")
    X = np.random.default_rng(2).standard_normal((4, g.dim))
    before = g.sigma(X)
    free = _free()
    release_memory()
    assert _free() - free >= 8 * (v * (v + 1) // 2) ** 2 + 4 * o * v**3  # pair integrals, FP32 coupling block
    assert np.abs(g.sigma(X) - before).max() <= 3e-5 * np.abs(before).max()
    g.close()


def test_digits_of_constants_are_given_back():
    """The digits that an FP64 handle keeps of its constant operands are memory held for speed too: they go back
    with the rest, and are made again by the next sigma.  At 10 / 120 each form of an o^2 v^2 constant is 23 MB;
    sigma keeps more than two.  FP64 bound 1e-11."""
    from paper_2012_06714_gb300 import ADC, release_memory

    s = make_system(10, 120, 200, seed=1)
    g = ADC(s.eps, s.B, 10, order=3, kind="ea", precision="fp64")
    X = np.random.default_rng(2).standard_normal((2, g.dim))
    before = g.sigma(X)
    release_memory()  # pair integrals and coupling block, which are not formed again, and the digits
    for _ in range(2):
        assert np.abs(g.sigma(X) - before).max() <= 1e-11 * np.abs(before).max()
        free = _free()
        release_memory()
        assert _free() - free >= 2 * 16 * (10 * 120) ** 2
    g.close()


def test_solves_with_graphs_that_run_out_of_memory_leave_nothing():
    """A solve with cuda_graphs that runs out of memory somewhere on its way to a captured sigma gives back that
    sigma's buffers (2 x 7 MB at these sizes): with no handle left the device has as much free memory as before,
    up to 8 MB."""
    from paper_2012_06714_gb300 import ADC, release_memory
    from paper_2012_06714_gb300._lib import ADCError

    o, v = 6, 160
    s = make_system(o, v, 40, seed=1)
    stream = torch.cuda.Stream()

    def solve(leave):
        g = ADC(s.eps, s.B, o, order=3, kind="ea", precision="bf16x3", cuda_graphs=1, max_iter=3)
        g.set_stream(stream.cuda_stream)
        release_memory()
        hold = torch.empty(_free() - leave, dtype=torch.uint8, device="cuda") if leave else None
        try:
            g.davidson(4, tol=1e-6)
            return True
        except ADCError as e:
            assert e.code == -2
            return False
        finally:
            del hold
            torch.cuda.empty_cache()
            g.close()

    assert solve(0)
    release_memory()
    free = _free()
    done = [solve(m << 20) for m in range(100, 2000, 100)]
    assert not all(done) and any(done)
    assert _free() >= free - (8 << 20)
