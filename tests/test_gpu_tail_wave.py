"""The shared-memory tail of the wave cycle, a thread holding several rows of a
column: levels at the edges of what a block takes (64 columns, 64 rows in
FP32, 32 in FP64), rows that do not fill a thread's share, tall and wide
levels, many levels, a sponge; without ADR corrections, so that only the wave
cycle runs.  Against one launch per pass and against the oracle, with the
tolerances of the cycle's other forms (FP64 1e-12, mixed 1e-5)."""
import numpy as np
import pytest

import synth
from gpu_util import cdt, rel, rnd
from oracle.cycle import CycleParams, Hierarchy
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "mixed": 1e-5}


# level 4 (an eighth): 64 x 64, 63 x 64, 32 x 31, 33 x 17, 64 x 9, 10 x 62, 31 x 31 down to 3
@pytest.mark.parametrize("n,ny,n_cmax", [(512, 517, 15), (511, 519, 15), (263, 250, 15), (264, 143, 15), (512, 79, 16),
                                         (87, 503, 15), (255, 255, 3)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_wave_tail(n, ny, n_cmax, prec):
    bc = "sponge" if n % 2 == 0 else "abc1"
    I = synth.config_layered_rect(n=n, ny=ny, omega=0.3 * (max(n, ny) + 1), bc=bc)
    g = rnd((ny, n), 3, cdt(prec))
    out, launches = {}, {}
    for tail in (64, 0):
        p = B.default_params(precision=prec, n_cmax=n_cmax, adr=0, tail_nmax=tail)
        h = B.mg_setup([(n, I.omega, I.k, I.phi, bc, ny)], p)
        u = np.zeros((ny, n), cdt(prec))
        B.mg_cycle(h, u, g, 1)
        out[tail], launches[tail] = u, B.mg_cycle_launches(h)
        B.mg_destroy(h)
    H = Hierarchy(n, I.k, I.phi, I.omega, bc, CycleParams(n_cmax=n_cmax, adr=False), ny=ny)
    ref = H.cycle(np.zeros((ny, n), np.complex128), g.astype(np.complex128))
    assert launches[64] < launches[0]
    assert rel(out[64], ref) < TOL[prec] and rel(out[0], ref) < TOL[prec]
