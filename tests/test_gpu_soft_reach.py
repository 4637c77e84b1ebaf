"""Support solves around the size of the neighbour list (144): targets below it,
at it and above it, from guesses that are right, half and twice the solution, and
mixed, so that a pass lists, sums while it records, and sums alone; against the
oracle (tolerances of test_gpu_soft)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_13792_gb300 import ics

from test_gpu_soft import gpu_solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ngb", [40.0, 83.0, 121.0, 144.0, 145.0, 260.0])
@pytest.mark.parametrize("factor", [1.0, 0.5, 2.0, 0.0])
@pytest.mark.parametrize("kind", [ics.plummer, ics.uniform_sphere])
def test_supports_around_the_lists_size(n_ngb, factor, kind):
    n = 1811
    pos, vel, mass = kind(n, seed=900)
    sol = O.soft_solve(pos, mass, 0.3, n_ngb=n_ngb, tol=1e-12, max_iter=200)
    assert sol["converged"]
    h0 = sol["h"] * (factor if factor > 0 else 2.0 ** ics.rng(901).uniform(-1, 1, n))
    ref = O.soft_solve(pos, mass, h0, n_ngb=n_ngb, tol=1e-12, max_iter=200)
    got = gpu_solve(pos, mass, h0, n_ngb, max_iter=200)
    assert ref["converged"] and got["flags"] == 0
    np.testing.assert_allclose(got["h"], ref["h"], rtol=1e-10, atol=0)
    np.testing.assert_allclose(got["omega"], ref["omega"], rtol=1e-8, atol=0)
    np.testing.assert_allclose(got["zeta"], ref["zeta"], rtol=1e-8, atol=0)


def test_guesses_beyond_the_range_of_fp32():
    """Every source is in reach of a guess of 1e39, and its FP32 value is infinite:
    the solve still ends, at the same supports."""
    n = 700
    pos, vel, mass = ics.uniform_sphere(n, seed=910)
    h0 = np.where(np.arange(n) % 2 == 0, 1e39, 0.5)
    ref = O.soft_solve(pos, mass, np.full(n, 0.5), n_ngb=32.0, tol=1e-12, max_iter=400)
    got = gpu_solve(pos, mass, h0, 32.0, max_iter=400)
    assert ref["converged"] and got["flags"] == 0
    np.testing.assert_allclose(got["h"], ref["h"], rtol=1e-10, atol=0)
