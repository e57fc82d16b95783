"""The update u += ||r|| Z y at the end of a restart (FP32: a compensated sum,
the vectors of Z loaded five at a time) at the lengths where its groups can go
wrong: one vector, a group less one, a group, one more, two groups, the longest
restart; against the FP64 handle.

The directions z_j of the two handles differ by less than 1e-5 (the bound of
the mixed cycle), so the minimal residual over at most 22 of them moves by less
than 22 * 1e-5 of ||g|| times the condition of the Hessenberg systems, taken as
5; a vector left out or taken twice changes it by several per cent."""
import numpy as np
import pytest

import synth
from gpu_util import lib_handle
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, 4, 5, 6, 10, 11, 22])
def test_update_matches_fp64(steps):
    insts = [synth.config_lognormal(n=n, omega=0.4 * (n + 1), seed=3 + n) for n in (47, 100)]
    g = np.concatenate([I.g.ravel() for I in insts])
    r = {}
    for prec in ("fp64", "mixed"):
        h = lib_handle(insts, prec, M=1, restart=22, tol=0.0, maxit=1 << 30, autotune=0)
        u = np.zeros_like(g)
        B.mg_solve_begin(h, u, g)
        B.mg_solve_steps(h, steps)
        r[prec] = B.mg_solve_end(h, u)
        B.mg_destroy(h)
    assert abs(r["mixed"] - r["fp64"]) < 22 * 1e-5 * 5
