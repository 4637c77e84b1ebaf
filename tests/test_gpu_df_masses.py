"""GRAV_F64, open boundaries, where a few terms carry a sum or the terms cancel,
so that nothing averages the rounding of a pair: one heavy element among light
ones (as target and as source), a stellar mass function, few elements, an a_bar
with one large row or of random signs.  The reference is in extended precision,
without softening (h below every separation).

Tolerance: a pair in FP64 is good to 4 or 5 units in its last place (5e-16; the
rsqrt, three products, the sums of three squares), the running sum of a tile adds
1.1e-16 sqrt(256 / 2) of its terms' root sum of squares, and a sum of positive
terms that many sources share may be 1e-15 of its magnitude off in two parts; the
largest of some hundred such errors is four times their rms.  So 7e-15 of the
root sum of squares of the terms, or 2e-15 of the sum of their magnitudes."""
import numpy as np
import pytest

from paper_2010_13792_gb300 import grav, ics

from gpu_util import run_eval
from test_gpu_backward import gpu_backward
from test_gpu_batched import run_batched

pytestmark = pytest.mark.gpu
L = np.longdouble
H = 1e-9
TOL, TOL_SUM = 7e-15, 2e-15


def _norm(x):
    return np.sqrt((x.astype(L) ** 2).sum(-1))


def _check(got, ref, size, rows, cancel=False):
    """got [rows, c] against the sums `ref` of terms whose norms are size[row] (list);
    cancel: of random signs, held to their root sum of squares alone."""
    for k in range(len(rows)):
        bound = TOL * np.sqrt((size[k] ** 2).sum())
        if not cancel:
            bound = max(bound, TOL_SUM * size[k].sum())
        e = _norm(np.atleast_1d(got[k] - ref[k]))
        assert e <= bound, (rows[k], float(e), float(bound))


def _forward(out, pos, vel, mass, rows):
    X, V, M = pos.astype(L), vel.astype(L), mass.astype(L)
    acc, tid, sa, st, jerk, sj = [], [], [], [], [], []
    for i in rows:
        k = np.ones(len(mass), bool)
        k[i] = False
        d, v, m = (X - X[i])[k], (V - V[i])[k], M[k]
        r2 = (d * d).sum(1)
        f = m / (r2 * np.sqrt(r2))
        g = f / r2
        acc.append((f[:, None] * d).sum(0))
        sa.append(np.abs(f) * np.sqrt(r2))
        jerk.append((f[:, None] * v - 3 * (g * (d * v).sum(1))[:, None] * d).sum(0))
        # (the sums run over velocities relative to a tile's: bounded by the largest)
        sj.append(4 * np.abs(f) * np.sqrt((v * v).sum(1)).max())
        t = [(g * d[:, a] * d[:, b]).sum() for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))]
        F = f.sum()
        tid.append([3 * t[0] - F, 3 * t[1] - F, 3 * t[2] - F, 3 * t[3], 3 * t[4], 3 * t[5]])
        st.append(6 * np.abs(f))
    _check(out["acc"][rows], np.array(acc), sa, rows)
    _check(out["tidal"][rows], np.array(tid), st, rows)
    _check(out["jerk"][rows], np.array(jerk), sj, rows)


def _rows(n, *extra):
    return np.unique(np.concatenate([np.linspace(0, n - 1, min(n, 20)).astype(int), np.array(extra, int)]))


@pytest.mark.parametrize("mu", [1e-2, 1e-4, 1e-6, 1e-9, 1e-12, 1e-15])
@pytest.mark.parametrize("n,split", [(300, 1), (2000, 1), (6001, 0), (9000, 0)])
def test_one_heavy_among_light(n, split, mu):
    pos, vel, mass = ics.uniform_sphere(n, seed=400 + n)
    mass = np.full(n, mu)
    mass[n // 2] = 1.0
    out = run_eval(pos, vel, mass, h=H, precision=grav.F64, max_split=split)
    _forward(out, pos, vel, mass, np.array([n // 2]))
    _forward(out, pos, vel, mass, _rows(n))


@pytest.mark.parametrize("decades", [3, 6, 14])
@pytest.mark.parametrize("n,split", [(257, 1), (1000, 1), (7000, 0)])
def test_spread_masses(n, split, decades):
    pos, vel, mass = ics.plummer(n, seed=410 + n)
    u = ics.rng(411).uniform(0, 1, n)
    # 3: the stellar mass function from 0.1 to 100
    mass = 0.1 * (1 - u * (1 - 1000 ** -1.35)) ** (-1 / 1.35) if decades == 3 else 10.0 ** (-decades * u)
    out = run_eval(pos, vel, mass, h=H, precision=grav.F64, max_split=split)
    _forward(out, pos, vel, mass, _rows(n, int(np.argmax(mass))))


@pytest.mark.parametrize("sizes", [(2, 3, 5, 33, 64), (128, 129, 200, 256, 257)])
def test_batched_systems_of_few(sizes):
    parts = [ics.plummer(n, seed=420 + n) for n in sizes]
    pos, vel, mass = (np.concatenate([p[c] for p in parts]) for c in range(3))
    off = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    out = run_batched(pos, vel, mass, np.stack([off, sizes], axis=1).astype(np.int64),
                      np.arange(mass.size, dtype=np.int32), H, grav.F64)
    for (p, v, m), o in zip(parts, off):
        _forward({k: x[o:o + m.size] for k, x in out.items()}, p, v, m, _rows(m.size))


def _adjoint(pos, mass, a_bar, split, rows, cancel=False):
    n = mass.size
    zero3, zero6, zero = np.zeros((n, 3)), np.zeros((n, 6)), np.zeros(n)
    pb, mb = gpu_backward(pos, mass, a_bar, 0.0, zero3, zero6, zero, H, grav.F64, max_split=split)
    X, A, M = pos.astype(L), a_bar.astype(L), mass.astype(L)
    p, m, sp, sm = [], [], [], []
    for i in rows:
        k = np.ones(n, bool)
        k[i] = False
        d, b = (X - X[i])[k], A[k]
        r2 = (d * d).sum(1)
        f = 1 / (r2 * np.sqrt(r2))
        da = (d * b).sum(1)
        p.append(M[i] * ((f[:, None] * b).sum(0) - (3 * f / r2 * da)[:, None].T.dot(d)[0]))
        m.append(-(f * da).sum())
        # (f a_bar and 3 f (d . a_bar) d / r^2, summed apart)
        sp.append(M[i] * f * np.sqrt((b * b).sum(1) + 9 * da * da / r2))
        sm.append(f * (np.abs(da) if cancel else np.sqrt(r2 * (b * b).sum(1))))
    _check(pb[rows], np.array(p), sp, rows, cancel)
    _check(mb[rows], np.array(m), sm, rows, cancel)


@pytest.mark.parametrize("mu", [1e-4, 1e-8, 1e-12])
@pytest.mark.parametrize("n,split", [(300, 1), (3000, 0), (6100, 0)])
def test_adjoint_one_large_row(n, split, mu):
    pos, vel, mass = ics.uniform_sphere(n, seed=430 + n)
    a_bar = np.full((n, 3), mu)
    a_bar[n // 2] = 1.0
    _adjoint(pos, mass, a_bar, split, np.array([n // 2]))
    _adjoint(pos, mass, a_bar, split, _rows(n))


@pytest.mark.parametrize("decades", [0, 6])
@pytest.mark.parametrize("n,split", [(300, 1), (3000, 0), (6100, 0)])
def test_adjoint_random_signs(n, split, decades):
    pos, vel, mass = ics.plummer(n, seed=440 + n)
    a_bar = ics.rng(441).normal(0, 1, (n, 3)) * 10.0 ** ics.rng(442).uniform(-decades, 0, (n, 1))
    _adjoint(pos, mass, a_bar, split, _rows(n), cancel=True)
