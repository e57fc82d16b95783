"""mg_eikonal ends when no value decreases by more than tol, also where tol is
less than a few units in the last place of tau (slowness 1e5, tau up to 1e5,
tol = 1e-12 against a unit of 1.5e-11): then no update may decrease its node at
all.

The update, computed in FP64 on the device, ends in a sum rounded to half a
unit of tau; before it, with f = s h: |a - b| <= f exact or to half a unit, 2 f^2
to half a unit and the difference of squares (>= f^2) to another, so the root
(<= 1.42 f) to 2.2e-16 of itself and the unit of its own rounding, the sum (<=
2.42 f) to half a unit, and the half of all this less than 4e-16 f.  A node that
rests because its update is not below its value lies no farther than that above
the exact update, formed here in extended precision."""
import numpy as np
import pytest

from paper_2404_02493_gb300 import binding as B

pytestmark = pytest.mark.gpu


def exact_update(tau, s, h):
    p = np.pad(tau.astype(np.longdouble), 1, constant_values=np.inf)
    a = np.minimum(p[1:-1, :-2], p[1:-1, 2:])
    b = np.minimum(p[:-2, 1:-1], p[2:, 1:-1])
    f = (s * h).astype(np.longdouble)
    d = np.abs(a - b)
    two = d < f
    root = np.sqrt(np.where(two, 2 * f * f - np.where(two, d, 0) ** 2, 0))
    return np.minimum(a, b) + np.where(two, 0.5 * (np.where(two, d, 0) + root), f)


@pytest.mark.parametrize("n,ny", [(64, 64), (127, 127), (301, 75)])
@pytest.mark.parametrize("scale,tol", [(1e5, 1e-12), (1e5, 0.0), (64.0, 1e-15)])
def test_no_value_decreases_by_more_than_tol(n, ny, scale, tol):
    h = 1.0 / (max(n, ny) + 1)
    s = scale * np.random.default_rng(n).uniform(1.0, 3.0, (ny, n))
    x0, y0 = 0.41 * (n + 1) * h, 0.27 * (ny + 1) * h
    tau = np.empty_like(s)
    st, _ = B.mg_eikonal_rect(n, ny, s, x0, y0, tau, tol=tol)
    assert st == B.MG_OK
    X, Y = np.meshgrid((np.arange(n) + 1) * h, (np.arange(ny) + 1) * h)
    free = np.hypot(X - x0, Y - y0) > 3.0 * h * (1 + 1e-12)
    above = tau - exact_update(tau, s, h)
    over = (above - (0.5 * np.spacing(tau) + 4e-16 * s * h))[free]
    assert over.max() <= 0, (above / np.spacing(tau))[free].max()
