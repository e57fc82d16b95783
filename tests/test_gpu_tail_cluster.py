"""The coarse ADR levels in one cluster launch per instance (automatic for one
instance; tail_nmax): whole corrections where the correction level fits, the
V-cycle below it elsewhere.  Sizes where the dealing of rows to blocks can go
wrong: fewer rows than blocks, even and odd sides, a last row of its own,
wide and tall levels, two levels and many, instances of different depth.

Against one launch per pass (tail_nmax = 0) and against the oracle, with the
tolerances of the cycle's other forms (FP64 1e-12, mixed 1e-5 per cycle)."""
import numpy as np
import pytest

import synth
from gpu_util import cdt, rel, rnd
from oracle.cycle import CycleParams, Hierarchy
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "mixed": 1e-5}


def instance(n, ny, bc):
    return synth.config_layered_rect(n=n, ny=ny, omega=0.3 * (max(n, ny) + 1), bc=bc)


def cycles(insts, shapes, prec, **kw):
    spec = [(I.n, I.omega, I.k, I.phi, I.bc, ny) for I, (_, ny) in zip(insts, shapes)]
    h = B.mg_setup(spec, B.default_params(precision=prec, M=2, **kw))
    g = [rnd((ny, n), 5 + n, cdt(prec)) for n, ny in shapes]
    u = np.zeros(sum(a.size for a in g), cdt(prec))
    B.mg_cycle(h, u, np.concatenate([a.ravel() for a in g]), 1)
    launches = B.mg_cycle_launches(h)
    B.mg_destroy(h)
    out, at = [], 0
    for a in g:
        out.append(u[at:at + a.size].reshape(a.shape))
        at += a.size
    return g, out, launches


# (n, ny, n_cmax): level 2 of 31, 63, 127 rows (whole corrections), even
# sides, ragged, tall, a last row of its own (129 = 8 * 16 + 1), two levels, six levels
@pytest.mark.parametrize("n,ny,n_cmax", [(63, 63, 15), (127, 127, 15), (255, 255, 15), (128, 128, 15), (100, 61, 15),
                                         (259, 131, 15), (131, 259, 15), (40, 200, 15), (66, 66, 32), (127, 127, 3)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_cluster_levels(n, ny, n_cmax, prec):
    bc = "sponge" if n % 2 == 0 else "abc1"
    I = instance(n, ny, bc)
    kw = dict(n_cmax=n_cmax, adr_bc="abc", autotune=0)
    g, u, lt = cycles([I], [(n, ny)], prec, tail_nmax=129, **kw)
    _, v, lp = cycles([I], [(n, ny)], prec, tail_nmax=0, **kw)
    H = Hierarchy(n, I.k, I.phi, I.omega, bc, CycleParams(n_cmax=n_cmax, M=2, adr_bc="abc"), ny=ny)
    ref = H.cycle(np.zeros((ny, n), np.complex128), g[0].astype(np.complex128))
    assert lt < lp
    assert rel(u[0], ref) < TOL[prec] and rel(v[0], ref) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_cluster_levels_of_a_batch(prec):
    """Clusters of instances that fit, per-level launches of those that do
    not, whole corrections of the small ones: one handle."""
    shapes = [(127, 127), (320, 319), (47, 90), (255, 100)]
    insts = [instance(n, ny, "abc1") for n, ny in shapes]
    g, u, lt = cycles(insts, shapes, prec, tail_nmax=63, autotune=0)
    for I, (n, ny), a, b in zip(insts, shapes, g, u):
        H = Hierarchy(n, I.k, I.phi, I.omega, I.bc, CycleParams(M=2), ny=ny)
        assert rel(b, H.cycle(np.zeros((ny, n), np.complex128), a.astype(np.complex128))) < TOL[prec]
