"""One launch for all Chebyshev steps of a small FP32 level, a region of 64 x
64 nodes in registers: 1 to 8 steps (tiles of 60 down to 32 columns), 9 steps
(the tile kernel), levels at the edge of one tile and one column past it, wide
and tall, more tiles than one row of them, the sponge term; against the FP64
oracle with the tolerance of the other FP32 Chebyshev passes (1e-5)."""
import numpy as np
import pytest

import synth
from gpu_util import rel, rnd
from oracle.cycle import CycleParams, Hierarchy
from oracle.smoothers import chebyshev
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


# level 2: 44 x 45, 64 x 31, 32 x 33, 35 x 150, 129 x 56, 97 x 97
@pytest.mark.parametrize("n,ny", [(89, 91), (129, 63), (64, 67), (71, 301), (258, 113), (195, 195)])
@pytest.mark.parametrize("q", [1, 2, 3, 5, 8, 9])
def test_cheb_region(n, ny, q):
    bc = "sponge" if n == 195 else "abc1"
    I = synth.config_layered_rect(n=n, ny=ny, omega=0.3 * (max(n, ny) + 1), bc=bc)
    p = B.default_params(precision="mixed", n_cmax=15, cheb_iters=q)
    h = B.mg_setup([(n, I.omega, I.k, I.phi, bc, ny)], p)
    H = Hierarchy(n, I.k, I.phi, I.omega, bc, CycleParams(n_cmax=15), ny=ny)
    for l in H.lam_max:
        shape = (B.mg_level_ny(h, 0, l), B.mg_level_n(h, 0, l))
        u, g = rnd(shape, 6, np.complex64), rnd(shape, 7, np.complex64)
        out = u.copy()
        B.mg_chebyshev(h, 0, l, out, g, q)
        b = H.lam_max[l]
        ref = chebyshev(H.lev(l), u.astype(np.complex128), g.astype(np.complex128), b / H.alpha[l], b, q)
        assert rel(out.astype(np.complex128), ref) < 1e-5, (l, rel(out, ref))
    B.mg_destroy(h)
