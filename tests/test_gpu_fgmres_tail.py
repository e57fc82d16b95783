"""The small dense work at the end of the two Gram-Schmidt passes (column
update, Givens rotations, back substitution: one row per lane of a warp) at
the restart lengths where it can go wrong, a restart included: 1, 2, 16, 17
and the longest, against the three-pass form, whose kernels do it in one
thread.

Both forms orthogonalise to working precision, so the iterates differ by the
working precision times the number of steps times the condition of the
Hessenberg systems, taken as 1e3 (eps 1.1e-16 or 6e-8, 23 steps)."""
import numpy as np
import pytest

import synth
from gpu_util import lib_handle, rel
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restart", [1, 2, 16, 17, 22])
@pytest.mark.parametrize("prec,tol", [("fp64", 23 * 1.1e-16 * 1e3), ("mixed", 23 * 6e-8 * 1e3)])
def test_two_pass_steps_match_three_pass(prec, tol, restart):
    insts = [synth.config_lognormal(n=n, omega=0.4 * (n + 1), seed=3 + n) for n in (47, 100)]
    g = np.concatenate([I.g.ravel() for I in insts])
    out = {}
    for passes in (2, 3):
        h = lib_handle(insts, prec, M=1, restart=restart, tol=0.0, maxit=1 << 30, fgmres_passes=passes, autotune=0)
        u = np.zeros_like(g)
        B.mg_solve_begin(h, u, g)
        B.mg_solve_steps(h, restart + 1)
        r = B.mg_solve_end(h, u)
        B.mg_destroy(h)
        out[passes] = (u, r)
    assert rel(out[2][0], out[3][0]) < tol
    assert abs(out[2][1] - out[3][1]) < tol
