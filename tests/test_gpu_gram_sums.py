"""The sums and the small solve that end a gram pass, at the sizes where they
can go wrong: a level that is one block (no partials), two blocks, ragged
tiles, more partials than a round of the last block takes; every candidate,
against GMRES(3) of the oracle (FP64, 1e-11 as for the other sizes) and, in
FP32, against the same sweep of the FP64 handle.

FP32 tolerance: the normal equations of three scaled basis vectors lose
cond(K)^2 eps32; with random right-hand sides on these levels cond(K)^2 is
below 1e2, so 1e2 * 32 * 6e-8 = 2e-4 covers the sums of every order."""
import numpy as np
import pytest

import synth
from gpu_util import rel, rnd
from oracle.cycle import CycleParams, Hierarchy
from oracle.operators import adr_apply
from oracle.smoothers import gmres
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cand", range(B.MG_TILE_CANDIDATES))
@pytest.mark.parametrize("n,ny,n_cmax", [(19, 15, 4), (66, 17, 15), (70, 35, 15), (130, 98, 15), (600, 520, 15)])
def test_gram_sums(cand, n, ny, n_cmax):
    I = synth.config_layered_rect(n=n, ny=ny, omega=0.3 * (max(n, ny) + 1))
    H = Hierarchy(n, I.k, I.phi, I.omega, I.bc, CycleParams(n_cmax=n_cmax, M=1), ny=ny)
    lev = H.lev(2)
    b = rnd((lev.rows, lev.n), 4)
    ref = gmres(lambda v: adr_apply(H.adr[2], v), b, None, 3)
    for prec, tol, dt in (("fp64", 1e-11, np.complex128), ("mixed", 2e-4, np.complex64)):
        p = B.default_params(precision=prec, n_cmax=n_cmax, M=1, tile_candidate=cand, autotune=0)
        h = B.mg_setup([(n, I.omega, I.k, I.phi, I.bc, ny)], p)
        for _ in range(2):   # the counters are back at zero for the next sweep
            x = np.zeros(b.shape, dt)
            B.mg_gmres3(h, 0, 2, b.astype(dt), x, 0)
            assert rel(x, ref) < tol, (prec, rel(x, ref))
        B.mg_destroy(h)
