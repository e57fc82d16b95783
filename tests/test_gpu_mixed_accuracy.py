"""What the compensated sums of the mixed form give, beyond its tolerances:
one cycle, and the residual after a restart, against the same in FP64, over
several media.

Measured over media of n = 100 to 700: error of a cycle 4.6e-7 .. 2.1e-6 (median
9e-7) with plain FP32 sums in the GMRES(3) sweeps and term-by-term Laplacians on
the small Chebyshev levels, 1.5e-7 .. 4.1e-7 (2.5e-7) with compensated sums, the
refined 3 x 3 solve and differences; residual after 20 steps with M = 2 off by
3e-6 .. 1e-5 of itself with a plain sum Z y and unrounded Hessenberg entries,
1e-8 .. 4e-7 now.  The bounds lie between the two (geometric mean: medians of the
cycle, ends of the ranges of the residual)."""
import numpy as np
import pytest

import synth
from gpu_util import cdt, lib_handle, rel, rnd
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


def test_error_of_a_cycle():
    err = []
    for n in (131, 199, 255, 310, 383, 447, 511, 600):
        I = synth.config_lognormal(n=n, omega=0.35 * (n + 1), seed=n)
        g = rnd((n, n), n, np.complex64)
        out = {}
        for prec in ("fp64", "mixed"):
            h = lib_handle([I], prec, M=2, autotune=0)
            u = np.zeros((n, n), cdt(prec))
            B.mg_cycle(h, u, g.astype(cdt(prec)), 1)
            B.mg_destroy(h)
            out[prec] = u.astype(np.complex128)
        err.append(rel(out["mixed"], out["fp64"]))
    assert np.median(err) < np.sqrt(9e-7 * 2.5e-7), err


@pytest.mark.parametrize("n", [255, 400, 511])
def test_residual_after_a_restart(n):
    I = synth.config_lognormal(n=n, omega=0.39 * (n + 1), seed=n)
    r = {}
    for prec in ("fp64", "mixed"):
        h = lib_handle([I], prec, M=2, tol=0.0, maxit=1 << 30, adr_bc="abc", autotune=0)
        u = np.zeros_like(I.g)
        B.mg_solve_begin(h, u, I.g)
        B.mg_solve_steps(h, 20)
        r[prec] = B.mg_solve_end(h, u)
        B.mg_destroy(h)
    assert abs(r["mixed"] - r["fp64"]) < np.sqrt(4e-7 * 3e-6) * r["fp64"], r
