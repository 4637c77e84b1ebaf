"""GRAV_F64, open boundaries, where lengths lie far apart: systems small against
their distance from the origin (FP64 positions there still resolve them), a tight
group among wide elements, units far from 1.  Every output has to stay finite
and as good as the sums allow.

Tolerance as in test_gpu_df: 2e-13 of the sum of the terms' magnitudes (a pair
is good to 2^-43 of itself); the tidal timestep is ||T||^(-1/2), so its relative
error is half that of the tidal norm."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2010_13792_gb300 import grav, ics

from gpu_util import DEV, T, run_eval, tidal_norm
from test_gpu_backward import gpu_backward
from test_gpu_batched import run_batched

pytestmark = pytest.mark.gpu
TOL = 2e-13


def _rows(n):
    return np.unique(np.linspace(0, n - 1, 48).astype(np.int32))


def _check(out, pos, vel, mass, rows, h):
    ref = O.eval_active(pos, vel, mass, rows, h=h)
    cond = O.conditioning(pos, vel, mass, rows, h=h)
    vmax = np.linalg.norm(vel - vel.mean(0), axis=1).max()
    for k in ("acc", "jerk", "tidal", "dt_grav"):
        assert np.all(np.isfinite(out[k][rows])), k
    assert np.all(np.linalg.norm(out["acc"][rows] - ref["acc"], axis=1) <= TOL * cond[:, 0])
    assert np.all(np.linalg.norm(out["jerk"][rows] - ref["jerk"], axis=1) <= 4 * TOL * vmax * cond[:, 2])
    dt = tidal_norm(out["tidal"][rows] - ref["tidal"])
    assert np.all(dt <= TOL * cond[:, 2])
    slack = TOL * cond[:, 2] / tidal_norm(ref["tidal"]) + 1e-15
    assert np.all(np.abs(out["dt_grav"][rows] / ref["dt_grav"] - 1.0) <= slack)


@pytest.mark.parametrize("offset", [1e8, 1e9, 1e10, 1e12])
@pytest.mark.parametrize("n,split", [(700, 1), (6001, 0), (9000, 0)])
def test_sphere_far_from_the_origin(offset, n, split):
    pos, vel, mass = ics.uniform_sphere(n, seed=300 + n)
    pos = pos + np.array([offset, -0.5 * offset, 0.25 * offset])
    out = run_eval(pos, vel, mass, h=1e-3, precision=grav.F64, max_split=split)
    _check(out, pos, vel, mass, _rows(n), 1e-3)


@pytest.mark.parametrize("width", [1e-6, 1e-8, 1e-10])
def test_tight_group_among_wide_elements(width):
    g = ics.rng(310)
    pos = np.concatenate([g.normal(0, 1, (5000, 3)), 0.7 + width * g.normal(0, 1, (400, 3))])
    pos = pos[ics.morton_order(pos)]
    n = pos.shape[0]
    vel, mass = g.normal(0, 1, (n, 3)), g.uniform(0.5, 1.5, n)
    out = run_eval(pos, vel, mass, h=1e-3 * width, precision=grav.F64)
    rows = np.unique(np.concatenate([_rows(n), np.argsort(np.linalg.norm(pos - 0.7, axis=1))[:24]])).astype(np.int32)
    _check(out, pos, vel, mass, rows, 1e-3 * width)


def test_batched_systems_far_apart():
    sizes, parts = (300, 700, 64), []
    for k, n in enumerate(sizes):
        pos, vel, mass = ics.uniform_sphere(n, seed=320 + k)
        parts.append((pos + 10.0 ** (9 + k), vel, mass))
    pos, vel, mass = (np.concatenate([p[c] for p in parts]) for c in range(3))
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    systems = np.stack([off, sizes], axis=1).astype(np.int64)
    out = run_batched(pos, vel, mass, systems, np.arange(mass.size, dtype=np.int32), 1e-3, grav.F64)
    for (p, v, m), o in zip(parts, off):
        own = {k: x[o:o + m.size] for k, x in out.items()}
        _check(own, p, v, m, _rows(m.size), 1e-3)


@pytest.mark.parametrize("offset", [1e9, 1e10, 1e12])
@pytest.mark.parametrize("n,split", [(700, 1), (3001, 0), (6100, 0)])
def test_gradient_far_from_the_origin(offset, n, split):
    h = 1e-3
    pos, vel, mass = ics.uniform_sphere(n, seed=330 + n)
    pos = pos + np.array([offset, -0.5 * offset, 0.25 * offset])
    a_bar = 1.0 + 0.3 * ics.rng(331).normal(0, 1, (n, 3))
    zero3, zero6, zero = np.zeros((n, 3)), np.zeros((n, 6)), np.zeros(n)
    rows = _rows(n)
    pb_o, mb_o = O.backward(pos, mass, a_bar, 0.0, zero3, zero6, zero, h=h, rows=rows)
    pb, mb = gpu_backward(pos, mass, a_bar, 0.0, zero3, zero6, zero, h, grav.F64, max_split=split)
    ab = np.linalg.norm(a_bar, axis=1)
    for k in rows:
        r = np.linalg.norm(pos - pos[k], axis=1)
        f = np.minimum(1.0 / np.maximum(r, 1e-100) ** 3, (32.0 / 3.0) / h ** 3)
        f[k] = 0.0
        assert np.linalg.norm(pb[k] - pb_o[k]) <= TOL * mass[k] * 4.0 * (f * ab).sum()
        assert abs(mb[k] - mb_o[k]) <= TOL * (f * r * ab).sum()
