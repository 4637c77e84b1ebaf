"""The adjoint on both sides of the line below which it keeps FP64 pair terms (half
a work item an SM), against the oracle, and the small ones no slower for an a_bar
that puts some sources of a tile in two parts and some in FP64 than for one that
puts all in FP64.  (They take the same time; both routes in a tile took 1.25 times as
long.  The line is half way.)

Tolerance: 2e-13 of the sum of the terms' magnitudes (test_gpu_df)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from gpu_util import DEV, T
from test_gpu_backward import gpu_backward
from test_gpu_df import TOL

pytestmark = pytest.mark.gpu


def _line():
    """The largest n whose items (128 targets x 128 sources) are at most half the SMs."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return 128 * int(np.sqrt(sms // 2))


@pytest.mark.parametrize("beyond", [-1, 0, 1, 130])
def test_either_side_of_the_line(beyond):
    n, h = _line() + beyond, 1e-3
    pos, vel, mass = ics.plummer(n, seed=700)
    a_bar = -pos * (1 + 0.3 * ics.rng(701).uniform(0, 1, (n, 1)))
    zero3, zero6, zero = np.zeros((n, 3)), np.zeros((n, 6)), np.zeros(n)
    pb_o, mb_o = O.backward(pos, mass, a_bar, 0.0, zero3, zero6, zero, h=h)
    pb, mb = gpu_backward(pos, mass, a_bar, 0.0, zero3, zero6, zero, h, grav.F64)
    ab = np.linalg.norm(a_bar, axis=1)
    for k in range(0, n, 17):
        r = np.linalg.norm(pos - pos[k], axis=1)
        f = np.minimum(1.0 / np.maximum(r, 1e-100) ** 3, (32.0 / 3.0) / h ** 3)
        f[k] = 0.0
        assert np.linalg.norm(pb[k] - pb_o[k]) <= TOL * mass[k] * 4.0 * (f * ab).sum()
        assert abs(mb[k] - mb_o[k]) <= TOL * (f * r * ab).sum()


def _best_ms(pos, mass, a_bar):
    n = mass.size
    P, M, A = T(pos), T(mass), T(a_bar)
    z3 = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    z6, z = torch.zeros(n, 6, dtype=torch.float64, device=DEV), torch.zeros(n, dtype=torch.float64, device=DEV)
    pb, mb = torch.zeros_like(z3), torch.zeros_like(z)
    p, ws, best = grav.params(h=1e-3, precision=grav.F64), grav.Workspace(), 1e9
    for k in range(30):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        grav.eval_backward(p, P, M, A, 0.0, z3, z6, z, pb, mb, workspace=ws)
        b.record()
        torch.cuda.synchronize()
        if k >= 5:
            best = min(best, a.elapsed_time(b))
    return best


def test_both_routes_cost_no_more_than_fp64():
    n = 500
    pos, vel, mass = ics.plummer(n, seed=710)
    both = -pos * (1 + 0.3 * ics.rng(711).uniform(0, 1, (n, 1)))
    assert _best_ms(pos, mass, both) <= 1.12 * _best_ms(pos, mass, ics.rng(712).normal(0, 1, (n, 3)))
