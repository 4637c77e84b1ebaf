"""Support solves with elements that have no place: a NaN or infinite position is
flagged, has no neighbours and is nobody's neighbour, and the other supports come
out as without it.  Sizes with and without padding in the last tile of 128, and
small enough that such an element's list would hold every source.  (Tolerances of
test_gpu_soft.)"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from test_gpu_soft import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf])
@pytest.mark.parametrize("n,where", [(60, 0), (100, 99), (128, 64), (130, 129), (1500, 700)])
def test_elements_without_a_place_touch_no_other(n, where, bad):
    pos, vel, mass = ics.uniform_sphere(n, seed=800 + n)
    pos[where, 1] = bad
    rest = np.arange(n) != where
    h0, n_ngb = 0.5, 16.0
    ref = O.soft_solve(pos[rest], mass[rest], h0, n_ngb=n_ngb, tol=1e-12, max_iter=60)
    got = gpu_solve(pos, mass, h0, n_ngb, max_iter=60)
    assert got["flags"] & grav.FLAG_NONFINITE
    assert ref["converged"]
    np.testing.assert_allclose(got["h"][rest], ref["h"], rtol=1e-10, atol=0)
    np.testing.assert_allclose(got["omega"][rest], ref["omega"], rtol=1e-8, atol=0)
    np.testing.assert_allclose(got["zeta"][rest], ref["zeta"], rtol=1e-8, atol=0)
    assert np.all(got["iters"][rest] >= 0)
    assert got["iters"][where] == -1 and got["flags"] & grav.FLAG_NOCONVERGE
