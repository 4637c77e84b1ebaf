"""The 128-thread kernel of small open-boundary evaluations (below 2^30
interactions) against the nominal configuration, on both sides of the line and
with the count on the host and on the device: the same tile sums, so the
results differ by the order in which the chunk partials are added, a few
units in the last place (held to 1e-13 of the target's own magnitudes)."""
import numpy as np
import pytest

from paper_2010_13792_gb300 import grav, ics

from gpu_util import run_eval

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(1, 1), (129, 129), (5000, 40), (40000, 26843), (40000, 26845),
                                 (40000, 700), (9000, 9000)])
@pytest.mark.parametrize("device_count", [True, False])
def test_few_against_nominal(n, m, device_count):
    pos, vel, mass = ics.plummer(n, seed=300 + n)
    idx = ics.active_subset(n, m / n, 301)
    nominal = grav.default_tile_config(grav.MIXED, idx.size)
    a = run_eval(pos, vel, mass, idx, h=0.01, precision=grav.MIXED, device_count=device_count)
    b = run_eval(pos, vel, mass, idx, h=0.01, precision=grav.MIXED, device_count=device_count,
                 tile_config=nominal)
    for k in ("acc", "jerk", "tidal", "pot"):
        x, y = a[k][idx].reshape(idx.size, -1), b[k][idx].reshape(idx.size, -1)
        scale = np.abs(y).max(axis=1, keepdims=True)
        assert np.all(np.abs(x - y) <= 1e-13 * scale), (k, np.abs(x - y).max())


def test_device_count_decides():
    """One index list, room for n targets, counts on both sides of the line."""
    import torch
    from gpu_util import T
    n = 40000
    pos, vel, mass = ics.uniform_sphere(n, seed=302)
    P, V, M = T(pos), T(vel), T(mass)
    idx = T(np.arange(n), torch.int32)
    out = {}
    for count in (1, 500, 26843, 26845, n):
        acc = torch.zeros(n, 3, dtype=torch.float64, device=P.device)
        jerk, tid = torch.zeros_like(acc), torch.zeros(n, 6, dtype=torch.float64, device=P.device)
        c = T(np.array([count]), torch.int32)
        grav.eval_active(grav.params(h=0.01), P, V, M, idx, c, n, acc, jerk, tid)
        out[count] = acc.cpu().numpy()
        assert np.all(out[count][count:] == 0) and np.all(np.abs(out[count][:count]).max(axis=1) > 0)
    full = out[n]
    for count, a in out.items():
        scale = np.abs(full[:count]).max(axis=1, keepdims=True)
        # (a warp's targets, so its near tiles, are the same except the last)
        whole = count // 32 * 32
        assert np.all(np.abs(a[:whole] - full[:whole]) <= 1e-13 * scale[:whole])
