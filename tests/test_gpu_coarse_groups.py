"""mg_setup where the memory for the matrices of all coarsest-level inverses at
once is not there (a stand-in for cudaMalloc that refuses sizes from a limit
on): it goes on with fewer at a time, down to one, with the same bits; where not
even one fits, MG_ENOMEM."""
import pytest

from fake_runtime import run

pytestmark = pytest.mark.gpu


def test_groups_shrink_to_what_is_free(tmp_path):
    out = run(tmp_path, """
        import numpy as np
        import synth
        from gpu_util import lib_handle, rnd
        from paper_2404_02493_gb300 import binding as B

        most = ctypes.c_size_t.in_dll(lib, "fake_malloc_max")
        refused = ctypes.c_long.in_dll(lib, "fake_mallocs_refused")
        # 12 operators of 256 nodes and 6 of 961: 2.1 and 29.7 MB of matrices each;
        # the handle's own allocations are below 24 MB
        insts = [synth.config_lognormal(n=n, omega=0.3 * (n + 1), seed=n) for n in (65, 63) for _ in range(6)]
        N = sum(I.n * I.n for I in insts)
        g = rnd((N,), 1)
        got = []
        for limit in (0, 140 << 20, 60 << 20, 32 << 20):
            most.value = limit
            r0 = refused.value
            h = lib_handle(insts, "fp64", M=1, n_cmax=31, autotune=0)
            most.value = 0
            assert (refused.value > r0) == (limit > 0)
            u = np.zeros_like(g)
            B.mg_cycle(h, u, g, 1)
            B.mg_destroy(h)
            got.append(u)
        assert all(np.array_equal(u, got[0]) for u in got[1:])
        most.value = 24 << 20
        try:
            lib_handle(insts, "fp64", M=1, n_cmax=31, autotune=0)
            raise SystemExit("not refused")
        except B.MgError as e:
            assert e.code == B.MG_ENOMEM
        most.value = 0
        print("passed")
    """)
    assert "passed" in out
