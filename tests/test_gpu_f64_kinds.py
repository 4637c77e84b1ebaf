"""The three kinds of open FP64 evaluation (FP64 pair terms for the smallest,
two-part FP32 on small and on large tiles) on both sides of the lines between
them, against the oracle within the FP64 path's stated bounds, and a workspace
sized for every target used with fewer."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from gpu_util import assert_f64, errors, run_eval

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(1, 1), (130, 130), (2176, 2176), (2177, 2177), (2816, 2816), (3073, 3073), (8192, 8191), (8193, 8193)])
def test_either_side_of_the_lines(n, m):
    pos, vel, mass = ics.plummer(n, seed=500 + n)
    idx = np.arange(m, dtype=np.int32)
    out = run_eval(pos, vel, mass, idx, h=1e-3, precision=grav.F64)
    if n == 1:
        assert np.all(out["acc"] == 0)
        return
    rows = np.unique(np.linspace(0, m - 1, 64).astype(np.int32))
    ref = O.eval_active(pos, vel, mass, rows, h=1e-3)
    assert_f64(errors(out, ref, rows))


def test_workspace_for_all_targets_does_for_few():
    n = 9001
    pos, vel, mass = ics.plummer(n, seed=77)
    p = grav.params(h=1e-3, precision=grav.F64, max_split=2)
    room = grav.lib().grav_eval_workspace_bytes(p, n, n)
    for m in (1, 500, 3000, n):
        assert grav.lib().grav_eval_workspace_bytes(p, n, m) <= room
