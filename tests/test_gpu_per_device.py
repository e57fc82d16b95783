"""Kernel attributes (the opt-in to more shared memory, to a cluster of 16 blocks)
hold on one device only: a handle on a second device sets them there as well.  A
stand-in names the only device differently for the second handle (host arrays)
and counts the calls; a third handle on either asks for nothing again."""
import pytest

from fake_runtime import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_second_device_gets_its_own_attributes(tmp_path, prec):
    out = run(tmp_path, """
        import numpy as np
        import synth
        from gpu_util import cdt, lib_handle, rnd
        from paper_2404_02493_gb300 import binding as B

        prec = %r
        I = synth.config_lognormal(n=527, omega=0.3 * 528, seed=3)
        g = rnd((527 * 527,), 1, cdt(prec))
        device = ctypes.c_int.in_dll(lib, "fake_device")
        calls = ctypes.c_long.in_dll(lib, "func_attributes")
        count = []
        for dev in (0, 1, 0, 1):
            device.value = dev
            c0 = calls.value
            for kw in (dict(autotune=0), dict(tail_nmax=0, cheb_iters=9)):
                h = lib_handle([I], prec, M=1, **kw)
                u = np.zeros_like(g)
                B.mg_cycle(h, u, g, 1)
                x = np.zeros(g.size, np.complex128)
                B.mg_solve_begin(h, x, I.g.ravel())
                B.mg_solve_steps(h, 1)
                B.mg_solve_end(h, x)
                if prec == "fp64":
                    B.mg_cycle_backward(h, 0 * g, g, 1, g, np.zeros(g.size), np.zeros(B.MG_MAX_LEVELS))
                B.mg_destroy(h)
            count.append(calls.value - c0)
        # (the setup of the inverses sets its one attribute on every call)
        each = count[2]
        assert count[0] > each + 10 and count[1] == count[0] and count[3] == each, count
        print("passed", count)
    """ % prec)
    assert "passed" in out
