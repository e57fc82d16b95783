"""mg_cycle_backward over more cycles than two, where the steps after the first
run one by one (several media, up to 3) or replay a captured step (one medium; 4
and more), on one medium and on two of different size: the gradients of K cycles are the sum of those of single
cycles, each from its own iterate and with the cotangent that the next cycle's
call gave.  The single calls run the same operations on the same values; only
the order in which the cycles' contributions to grad_phi and the weights are
added differs (K eps of their sum, taken as 1e-12 relative)."""
import numpy as np
import pytest

import synth
from fake_runtime import run
from gpu_util import lib_handle, rel, rnd
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(63,), (47, 95)])
@pytest.mark.parametrize("K", [3, 4, 5])
def test_gradients_of_many_cycles(sizes, K):
    insts = [synth.config_lognormal(n=n, omega=0.3 * (n + 1), seed=n) for n in sizes]
    N, W = sum(n * n for n in sizes), B.MG_MAX_LEVELS * len(sizes)
    h = lib_handle(insts, "fp64", M=2, n_cmax=7, autotune=0)
    g, ubar, u = rnd((N,), 1), rnd((N,), 2), rnd((N,), 3)
    gphi, gw, gu = np.zeros(N), np.zeros(W), np.zeros(N, complex)
    B.mg_cycle_backward(h, u, g, K, ubar, gphi, gw, gu)
    it = [u]
    for _ in range(K - 1):
        it.append(it[-1].copy())
        B.mg_cycle(h, it[-1], g, 1)
    rphi, rw, bar = np.zeros(N), np.zeros(W), ubar
    for uk in reversed(it):
        nxt = np.zeros(N, complex)
        B.mg_cycle_backward(h, uk, g, 1, bar, rphi, rw, nxt)
        bar = nxt
    B.mg_destroy(h)
    assert rel(gu, bar) < 1e-12
    assert rel(gphi, rphi) < 1e-12
    assert rel(gw, rw) < 1e-12


@pytest.mark.parametrize("which", [1, 2, 3])
def test_steps_are_emitted_where_the_capture_fails(tmp_path, which):
    """(a stand-in for the failing call, on the host)"""
    out = run(tmp_path, """
        import numpy as np
        import synth
        from gpu_util import lib_handle, rnd
        from paper_2404_02493_gb300 import binding as B

        insts = [synth.config_lognormal(n=n, omega=0.3 * (n + 1), seed=n) for n in (47, 63)]
        N = sum(I.n * I.n for I in insts)
        h = lib_handle(insts, "fp64", M=2, n_cmax=7, autotune=0)
        fake = ctypes.c_int.in_dll(lib, "fake_capture")
        refused = ctypes.c_int.in_dll(lib, "fake_captures_refused")

        def gradients():
            gphi, gw, gu = np.zeros(N), np.zeros(2 * B.MG_MAX_LEVELS), np.zeros(N, complex)
            B.mg_cycle_backward(h, rnd((N,), 3), rnd((N,), 1), 4, rnd((N,), 2), gphi, gw, gu)
            return gphi, gw, gu

        want = gradients()
        assert refused.value == 0
        fake.value = %d
        got = gradients()
        fake.value = 0
        assert refused.value == 2
        assert all(np.array_equal(a, b) for a, b in zip(want, got))
        B.mg_destroy(h)
        print("passed")
    """ % which)
    assert "passed" in out
