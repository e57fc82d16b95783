"""The automatic coarse tail serves handles of as many instances as clusters run
on the GPU at once, and none where none can be placed (a stand-in gives their
number); the cycle is the per-level one otherwise, launch by launch."""
import pytest

from fake_runtime import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("slots", [0, 3])
def test_tail_for_the_clusters_that_run_at_once(tmp_path, prec, slots):
    out = run(tmp_path, """
        import numpy as np
        import synth
        from gpu_util import cdt, lib_handle, rel, rnd
        from paper_2404_02493_gb300 import binding as B

        prec, slots = %r, %d
        ctypes.c_int.in_dll(lib, "fake_clusters").value = slots
        for ni in (1, 3, 4):
            # level 4 of n = 127 is the coarsest: there is no tail but the ADR one
            insts = [synth.config_lognormal(n=127, omega=30.0, seed=b) for b in range(ni)]
            g = rnd((sum(I.n * I.n for I in insts),), 1, cdt(prec))
            got = []
            for kw in (dict(), dict(tail_nmax=0)):
                h = lib_handle(insts, prec, M=2, autotune=0, **kw)
                u = np.zeros_like(g)
                B.mg_cycle(h, u, g, 1)
                got.append((B.mg_cycle_launches(h), u))
                B.mg_destroy(h)
            (la, ua), (lp, up) = got
            assert (la < lp) if ni <= slots else (la == lp), (ni, la, lp)
            assert rel(ua, up) < (1e-12 if prec == "fp64" else 1e-5)
        print("passed")
    """ % (prec, slots))
    assert "passed" in out
