"""The open-boundary FP64 kernels (two-part FP32 pair sums, listed pairs in
FP64) against the oracle where their tiling and ranges can go wrong: partial
sub-blocks and tiles, both tile sizes, masses and a_bar spread over six decades,
units far from 1, systems far from the origin, coincident elements, supports
from none to wider than the system.

Tolerance: a pair comes out within 2^-43 of itself (the two-part rounding, a
dozen operations of 2^-47), so a sum is held to 2e-13 of the sum of its terms'
magnitudes (oracle_conditioning)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from gpu_util import run_eval, tidal_norm
from test_gpu_backward import gpu_backward

pytestmark = pytest.mark.gpu
TOL = 2e-13


def _clustered(n, seed, shift):
    g = ics.rng(seed)
    pos = g.normal(0, 1, (n, 3)) * np.exp(g.uniform(-3, 1, (n, 1)))
    if n > 40:
        pos[n // 2: n // 2 + 3] = pos[n // 3]          # coincident elements
    pos = pos[ics.morton_order(pos)] + shift
    return pos, g.normal(0, 1, (n, 3)) + 5.0 * shift, 10.0 ** g.uniform(-6, 0, n)


@pytest.mark.parametrize("n", [2, 31, 33, 129, 257, 1000, 6001])
@pytest.mark.parametrize("h,shift,unit", [(1e-6, 0.0, 1.0), (0.05, 100.0, 1.0), (0.3, 0.0, 3e19),
                                          (50.0, 0.0, 1.0)])
def test_sums_vs_oracle(n, h, shift, unit):
    pos, vel, mass = _clustered(n, 90 + n, shift)
    pos, h, mass = pos * unit, h * unit, mass * unit ** 2
    idx = np.arange(n, dtype=np.int32) if n < 3000 else ics.active_subset(n, 0.1, 91)
    ref = O.eval_active(pos, vel, mass, idx, h=h)
    cond = O.conditioning(pos, vel, mass, idx, h=h)
    for split in (0, 1):                               # fine and coarse tiles for the small n
        out = run_eval(pos, vel, mass, idx, h=h, precision=grav.F64, max_split=split)
        assert np.all(np.linalg.norm(out["acc"][idx] - ref["acc"], axis=1) <= TOL * cond[:, 0])
        # (the jerk's sums run over tile-relative velocities: their magnitudes
        # are bounded by the largest relative velocity)
        vmax = np.linalg.norm(vel - vel.mean(0), axis=1).max()
        trace = cond[:, 2]
        assert np.all(np.linalg.norm(out["jerk"][idx] - ref["jerk"], axis=1) <= 4 * TOL * vmax * trace)
        assert np.all(tidal_norm(out["tidal"][idx] - ref["tidal"]) <= TOL * cond[:, 2])
        assert np.all(np.abs(out["pot"][idx] - ref["pot"]) <= TOL * np.abs(ref["pot"]))


@pytest.mark.parametrize("n", [33, 300, 6001])
@pytest.mark.parametrize("h", [1e-3, 0.5])
def test_adjoint_vs_oracle(n, h):
    pos, vel, mass = _clustered(n, 190 + n, 0.0)
    g = ics.rng(191)
    a_bar = g.normal(0, 1, (n, 3)) * 10.0 ** g.uniform(-6, 0, (n, 1))
    zero3, zero6, zero = np.zeros((n, 3)), np.zeros((n, 6)), np.zeros(n)
    pb_o, mb_o = O.backward(pos, mass, a_bar, 0.0, zero3, zero6, zero, h=h)
    # magnitudes of the pair terms: |f a_bar| + |g (d.a_bar) d| <= 4 f |a_bar| with
    # f <= r^-3, bounded inside the support by its central value
    rows = np.arange(n) if n < 3000 else np.arange(0, n, 37)
    big_p, big_m = np.zeros(rows.size), np.zeros(rows.size)
    ab = np.linalg.norm(a_bar, axis=1)
    for q, k in enumerate(rows):
        r = np.linalg.norm(pos - pos[k], axis=1)
        f = np.minimum(1.0 / np.maximum(r, 1e-300) ** 3, (32.0 / 3.0) / h ** 3)
        f[k] = 0.0
        big_p[q] = mass[k] * 4.0 * (f * ab).sum()
        big_m[q] = (f * r * ab).sum()
    for split in (0, 1):
        pb, mb = gpu_backward(pos, mass, a_bar, 0.0, zero3, zero6, zero, h, grav.F64, max_split=split)
        assert np.all(np.linalg.norm(pb - pb_o, axis=1)[rows] <= TOL * big_p)
        assert np.all(np.abs(mb - mb_o)[rows] <= TOL * big_m)
