"""GRAV_F64, open boundaries: the jerk of a smooth flow.  Neighbours of a turbulent
cloud move alike, so a close pair's velocities have to be subtracted before they
are weighted: in sums over a tile's velocities its large terms cancel.  Sizes with
listed pairs and with sub-blocks that are summed whole.  (The FP64 kernel of the
smallest evaluations sums over a tile's velocities, as it always did.)

Tolerance: over the targets, the rms of the error is at most 2e-15 of the rms of
the jerk: FP64 pairs with exact differences are good to 5e-16, two-part terms to
8e-15 with 64 and more of them to a tile (1e-15)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from gpu_util import run_eval

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,frac", [(3300, 1.0), (6794, 1.0), (16384, 0.1)])
def test_jerk_of_a_turbulent_cloud(n, frac):
    pos, vel, mass = ics.turbulent_cloud(n, seed=950)
    idx = np.arange(n, dtype=np.int32) if frac == 1.0 else ics.active_subset(n, frac, 951)
    out = run_eval(pos, vel, mass, idx, h=0.002, precision=grav.F64)
    ref = O.eval_active(pos, vel, mass, idx, h=0.002)
    for k in ("acc", "jerk", "tidal"):
        e = np.sqrt(((out[k][idx] - ref[k]) ** 2).sum() / (ref[k] ** 2).sum())
        assert e <= 2e-15, (k, e)
