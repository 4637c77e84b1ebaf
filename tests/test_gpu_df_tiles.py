"""Both tilings of the two-part FP64 force sums (tiles of the configuration's
sources below 2^26 pairs, of twice as many above) with sources split over several
items, in every configuration, on inputs that try them: a clustered system with
coincident elements, masses over six decades, far shifts and other units, supports
from none to wider than the system.  The sizes follow the number of SMs, so that
neither tiling gives way to the FP64 pairs of the smallest evaluations.

Tolerance: 2e-13 of the sum of the terms' magnitudes (test_gpu_df)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from gpu_util import run_eval, tidal_norm
from test_gpu_df import TOL, _clustered

pytestmark = pytest.mark.gpu


def _fine_n(threads, sources):
    """Elements whose items (blocks of `threads` x tiles of `sources`) pass 20 per
    SM, more than may be resident with the round after them."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return int(np.ceil(np.sqrt(20 * sms * threads * sources))) + 37


@pytest.mark.parametrize("cfg", [0, 1, 2])
@pytest.mark.parametrize("coarse", [False, True])
@pytest.mark.parametrize("h,shift,unit", [(1e-6, 0.0, 1.0), (0.05, 100.0, 1.0), (0.3, 0.0, 3e19),
                                          (50.0, 0.0, 1.0)])
def test_both_tilings(cfg, coarse, h, shift, unit):
    info = grav.tile_configs(grav.F64)[cfg]
    n = max(8193, 8192 + 64 * cfg + 33) if coarse else _fine_n(info["threads"], info["sources_per_tile"])
    assert (n * n >= 1 << 26) == coarse
    pos, vel, mass = _clustered(n, 600 + cfg, shift)
    pos, h, mass = pos * unit, h * unit, mass * unit ** 2
    rows = np.unique(np.concatenate([np.linspace(0, n - 1, 80).astype(int), np.arange(n // 2 - 2, n // 2 + 5)]))
    rows = rows.astype(np.int32)
    ref = O.eval_active(pos, vel, mass, rows, h=h)
    cond = O.conditioning(pos, vel, mass, rows, h=h)
    out = run_eval(pos, vel, mass, h=h, precision=grav.F64, tile_config=cfg)
    vmax = np.linalg.norm(vel - vel.mean(0), axis=1).max()
    assert np.all(np.linalg.norm(out["acc"][rows] - ref["acc"], axis=1) <= TOL * cond[:, 0])
    assert np.all(np.linalg.norm(out["jerk"][rows] - ref["jerk"], axis=1) <= 4 * TOL * vmax * cond[:, 2])
    assert np.all(tidal_norm(out["tidal"][rows] - ref["tidal"]) <= TOL * cond[:, 2])
    assert np.all(np.abs(out["pot"][rows] - ref["pot"]) <= TOL * np.abs(ref["pot"]))
