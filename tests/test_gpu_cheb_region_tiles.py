"""The one-launch smoothing of small FP32 levels where blocks take several tiles
(level 2 of 550 x 550 and 900 x 301 nodes: 169 and more tiles of 60 down to 32
columns for 152 SMs) and in its four-row form at the default five steps; against
the FP64 oracle with the tolerance of the other FP32 Chebyshev passes (1e-5)."""
import numpy as np
import pytest

import synth
from gpu_util import rel, rnd
from oracle.cycle import CycleParams, Hierarchy
from oracle.smoothers import chebyshev
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ny", [(1100, 1100), (1801, 603)])
def test_blocks_with_several_tiles(n, ny):
    I = synth.config_layered_rect(n=n, ny=ny, omega=0.3 * (max(n, ny) + 1))
    H = Hierarchy(n, I.k, I.phi, I.omega, I.bc, CycleParams(n_cmax=15), ny=ny)
    for q in (1, 2, 5, 6, 8):
        h = B.mg_setup([(n, I.omega, I.k, I.phi, I.bc, ny)], B.default_params(precision="mixed", cheb_iters=q, autotune=0))
        shape = (B.mg_level_ny(h, 0, 2), B.mg_level_n(h, 0, 2))
        u, g = rnd(shape, 6, np.complex64), rnd(shape, 7, np.complex64)
        out = u.copy()
        B.mg_chebyshev(h, 0, 2, out, g, q)
        B.mg_destroy(h)
        b = H.lam_max[2]
        ref = chebyshev(H.lev(2), u.astype(np.complex128), g.astype(np.complex128), b / H.alpha[2], b, q)
        assert rel(out.astype(np.complex128), ref) < 1e-5, (q, rel(out, ref))
