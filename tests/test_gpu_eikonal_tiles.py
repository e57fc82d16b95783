"""The tiled sweeps of mg_eikonal on media that send fronts through every tile
from every side."""
import numpy as np
import pytest

import oracle.eikonal as oeik
from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ny", [(31, 64), (65, 32), (64, 64), (97, 33)])
@pytest.mark.parametrize("src", [(0.02, 0.03), (0.41, 0.27), (0.97, 0.3)])
def test_eikonal_rough_medium_at_tile_edges(n, ny, src):
    """Slowness without any smoothness (uniform in [1, 3] per node: fronts
    from every side in every tile) on whole and ragged tiles: the oracle's
    fixed point to 8 ulp of max tau, as for the smooth media."""
    h = 1.0 / (max(n, ny) + 1)
    s = np.random.default_rng(n * ny).uniform(1.0, 3.0, (ny, n))
    x0, y0 = src[0] * (n + 1) * h, src[1] * (ny + 1) * h
    ref = oeik.eikonal(s, x0, y0, tol=0.0)
    tau = np.empty_like(s)
    st, _ = B.mg_eikonal_rect(n, ny, s, x0, y0, tau, tol=0.0)
    assert st == B.MG_OK
    assert np.max(np.abs(tau - ref)) <= 8 * np.spacing(ref.max())
