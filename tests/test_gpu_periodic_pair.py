"""The paired per-pair wrapping loop of the periodic mixed kernels at odd and
ragged source counts, with softened pairs in the even and the odd slot of a
source pair and across the faces of the box, against the oracle within the
mixed path's stated bounds, and the scalar layout within the same."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from gpu_util import assert_mixed, errors
from test_gpu_periodic import run_periodic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg", [0, 11])  # scalar layout, paired layout
@pytest.mark.parametrize("n,L", [(2, 1.0), (3, 0.3), (255, 1.0), (257, 0.3), (513, 1.0)])
def test_paired_wrapping_loop(n, L, cfg):
    g = ics.rng(400 + n)
    pos = g.uniform(0.0, L, (n, 3))
    h = 0.02 * L
    for i in range(4, n - 3, 5):  # neighbours at 0.4 h: even and odd slots in turn
        pos[i + 1] = pos[i] + 0.4 * h / np.sqrt(3.0)
    if n > 8:
        pos[0], pos[3] = [0.1 * h, 0.5 * L, 0.3 * L], [L - 0.2 * h, 0.5 * L, 0.3 * L]
    pos = np.mod(pos, L)
    vel, mass = g.normal(0.0, 1.0, (n, 3)), g.uniform(0.5, 1.5, n) / n
    ref = O.eval_active(pos, vel, mass, h=h, box=L)
    out = run_periodic(pos, vel, mass, None, h, L, grav.MIXED, tile_config=cfg)
    assert_mixed(errors(out, ref, np.arange(n)))
