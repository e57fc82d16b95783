"""A device allocation that fails ends the call with MG_ENOMEM before anything
is launched on it: every workspace limit below a handle's need (the allocation
that meets it differs), launch tables (built on first use; a limit that
mg_setup met does not count them), vectors of the adjoint.  The allocations
fail on the host, by the limit or by a stand-in for cudaMalloc."""
import numpy as np
import pytest

import synth
from fake_runtime import run
from gpu_util import cdt, lib_handle, rnd
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


def instances(prec):
    insts = [synth.config_lognormal(n=n, omega=0.3 * (n + 1), seed=n) for n in ((95,) if prec == "mixed" else (47, 63))]
    for I in insts:
        I.bc = "sponge" if I.n == 47 else "abc1"
    return insts


@pytest.mark.parametrize("prec,kw", [("mixed", {}), ("fp64", {}), ("mixed", dict(ray=1, M=3))])
def test_every_limit_below_the_need(prec, kw):
    insts = instances(prec)
    p = dict(n_cmax=7, autotune=0, **kw)
    N = sum(I.n * I.n for I in insts)
    g = rnd((N,), 1, cdt(prec))
    h = lib_handle(insts, prec, **p)
    need = B.mg_workspace_bytes(h)
    want = np.zeros_like(g)
    B.mg_cycle(h, want, g, 1)
    B.mg_destroy(h)
    for limit in sorted(set(np.linspace(1, need - 1, 60).astype(int))):
        with pytest.raises(B.MgError) as e:
            lib_handle(insts, prec, workspace_limit=int(limit), **p)
        assert e.value.code == B.MG_ENOMEM
    h = lib_handle(insts, prec, workspace_limit=need, **p)
    u = np.zeros_like(g)
    B.mg_cycle(h, u, g, 1)
    B.mg_destroy(h)
    assert np.array_equal(u, want)


def test_failing_allocations_of_later_calls(tmp_path):
    out = run(tmp_path, """
        import numpy as np
        import synth
        from gpu_util import lib_handle, rnd
        from paper_2404_02493_gb300 import binding as B

        after = ctypes.c_long.in_dll(lib, "fake_malloc_after")
        least = ctypes.c_size_t.in_dll(lib, "fake_malloc_min")
        insts = [synth.config_lognormal(n=n, omega=0.3 * (n + 1), seed=n) for n in (47, 63)]
        N = sum(I.n * I.n for I in insts)
        g, b = rnd((N,), 1), np.concatenate([I.g.ravel() for I in insts])
        kw = dict(M=1, n_cmax=7, autotune=0)

        def refused(call):
            # fail the first allocation of the call, then the second, ... until it passes
            k = 0
            while True:
                after.value = k
                try:
                    call()
                    after.value = -1
                    return k
                except B.MgError as e:
                    assert e.code == B.MG_ENOMEM, str(e)
                    after.value = -1
                    k += 1

        h = lib_handle(insts, "fp64", **kw)
        want = np.zeros_like(g)
        B.mg_cycle(h, want, g, 1)
        B.mg_destroy(h)
        h = lib_handle(insts, "fp64", **kw)
        tried = 0
        u = np.zeros_like(g)
        tried += refused(lambda: B.mg_cycle(h, u, g, 1))
        u[:] = 0
        B.mg_cycle(h, u, g, 1)
        assert np.array_equal(u, want)
        x = np.zeros_like(b)
        tried += refused(lambda: B.mg_solve_begin(h, x, b))
        B.mg_destroy(h)
        assert tried > 0
        # the adjoint's vectors: every fifth allocation
        h = lib_handle(insts, "fp64", **kw)
        B.mg_cycle(h, u, g, 1)
        def back(K, k):
            gp, gw = np.zeros(N), np.zeros(2 * B.MG_MAX_LEVELS)
            after.value = k
            try:
                B.mg_cycle_backward(h, g * 0, g, K, g, gp, gw)
                return gp, after.value
            except B.MgError as e:
                assert e.code == B.MG_ENOMEM, str(e)
            finally:
                after.value = -1
        for K in (1, 4):
            full, left = back(K, 100000)
            total = 100000 - left
            for k in range(0, total, 5):
                assert back(K, k) is None
            assert np.array_equal(back(K, -1)[0], full)
        B.mg_destroy(h)
        print("passed", tried, total)
    """)
    assert "passed" in out
