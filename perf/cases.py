"""Timing cases: the calls a user of the library makes, over the sizes and options in use.

A case is a dict of plain values.  ``listed()`` names twelve of them, ``draw`` gives more of the
same ranges, ``prepare`` makes what the calling program already holds (device arrays, indices,
workspaces, a captured graph), ``run`` makes one pass through the public entry points and returns
everything it computed, ``exact`` is the same result from plain FP64 tensor operations and ``work``
the bytes and operations that no implementation can do without.

Kinds:
  forces     one evaluation of a, j, T (and Phi, dt_grav) at a due set or at every element
  batched    the same over many independent systems in one call
  adjoint    accelerations and potential energy, then the gradient of a loss on both
  soft       per-element supports solved from guesses, then the forces with them
  tree       oct-tree build and walk
  bookkeep   one tick's selection, compaction, prediction and binning (no force sums)
  cycle      one captured cycle of block-timestep ticks of the adaptive integrator
"""
from __future__ import annotations

import math

import torch

from paper_2010_13792_gb300 import grav
from paper_2010_13792_gb300.adaptive import AdaptiveIntegrator
from paper_2010_13792_gb300.autograd import gravity

F64 = torch.float64
ETA = 0.01
K_MAX, DT_MAX = 6, 2.0 ** -4
PAIR_FLOPS, POT_FLOPS, ADJOINT_FLOPS = 56, 1, 31   # per interaction, an FMA counted as two
PRECISION = {"mixed": grav.MIXED, "f64": grav.F64}


def listed():
    return [
        # a small star cluster, every element a target: a few launches of some tens of microseconds
        {"name": "sphere 4096 mixed", "kind": "forces", "ic": "sphere", "n": 4096, "frac": 1.0,
         "precision": "mixed", "pot": False, "h": 0.01},
        # a substep of the adaptive scheme: 2% of a Plummer sphere is due, the count on the device
        {"name": "plummer 2^17 2% mixed", "kind": "forces", "ic": "plummer", "n": 131072,
         "frac": 0.02, "precision": "mixed", "pot": False, "h": 1e-3},
        # a full evaluation of a turbulent cloud with the potential (start of a run, energy check)
        {"name": "cloud 200003 mixed pot", "kind": "forces", "ic": "cloud", "n": 200003,
         "frac": 1.0, "precision": "mixed", "pot": True, "h": 2e-3},
        # the same in FP64, as energy() and predictor_error() evaluate it
        {"name": "plummer 2^16 f64", "kind": "forces", "ic": "plummer", "n": 65536, "frac": 1.0,
         "precision": "f64", "pot": False, "h": 1e-3},
        # the periodic pancake lattice, every element a target
        {"name": "pancake 40^3 mixed", "kind": "forces", "ic": "pancake", "n": 64000, "frac": 1.0,
         "precision": "mixed", "pot": False, "h": 2e-3},
        # many star clusters of uneven sizes and due sets advanced together
        {"name": "batch of 64 mixed", "kind": "batched", "n_sys": 64, "n_min": 512, "n_max": 16384,
         "precision": "mixed", "pot": False, "h": 0.01},
        # a training step: gradients of sum w |a|^2 + W with respect to positions and masses
        {"name": "adjoint 2^16 mixed", "kind": "adjoint", "ic": "plummer", "n": 65536,
         "precision": "mixed", "h": 1e-3},
        # the same in FP64 at a ragged size, as a gradient check runs it
        {"name": "adjoint 12289 f64", "kind": "adjoint", "ic": "sphere", "n": 12289,
         "precision": "f64", "h": 0.01},
        # fully adaptive softening: supports from guesses, then forces with the correction term
        {"name": "soft 40961 mixed", "kind": "soft", "ic": "cloud", "n": 40961,
         "precision": "mixed", "pot": False, "h": 0.06},
        # the tree solver on a cloud too large to sum directly every step
        {"name": "tree 2^18 mixed", "kind": "tree", "ic": "cloud", "n": 262144, "precision": "mixed",
         "pot": False, "h": 2e-3, "leaf": 8},
        # a tick's bookkeeping at the size of the headline cloud, odd
        {"name": "bookkeep 2^20+3", "kind": "bookkeep", "n": 1048579, "q_f": 0.5},
        # the adaptive integrator of a cluster: one captured cycle of ticks replayed
        {"name": "cycle 8192 mixed", "kind": "cycle", "ic": "plummer", "n": 8192, "k_max": 4,
         "precision": "mixed", "h": 1e-2, "q_f": 0.25},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes spread over the logarithm of the range (odd ones as they
    come), both precisions, due fractions from 1% to all, open and periodic boxes."""
    kind = rng.choice(["forces", "forces", "forces", "batched", "adjoint", "soft", "tree",
                       "bookkeep", "cycle"])
    precision = rng.choice(["mixed", "f64"])
    ic = rng.choice(["sphere", "plummer", "cloud"])
    h = {"sphere": 0.01, "plummer": 1e-3, "cloud": 2e-3}[ic]
    pot = rng.random() < 0.3
    if kind == "forces":
        if rng.random() < 0.2:
            n = _log_int(rng, 10, 40 if precision == "mixed" else 24) ** 3
            return {"kind": kind, "ic": "pancake", "n": n, "frac": 1.0, "precision": precision,
                    "pot": pot, "h": 2e-3}
        frac = rng.choice([1.0, round(math.exp(rng.uniform(math.log(0.01), 0.0)), 4)])
        top = min(1 << 20, int(math.sqrt((3.5e10 if precision == "mixed" else 3.5e9) / frac)))
        return {"kind": kind, "ic": ic, "n": _log_int(rng, 500, top), "frac": frac,
                "precision": precision, "pot": pot, "h": h}
    if kind == "batched":
        n_max = rng.choice([2048, 8192, 16384])
        return {"kind": kind, "n_sys": _log_int(rng, 3, 64), "n_min": 512,
                "n_max": n_max if precision == "mixed" else 8192, "precision": precision,
                "pot": pot, "h": 0.01}
    if kind == "adjoint":
        return {"kind": kind, "ic": ic, "n": _log_int(rng, 1000, 65536 if precision == "mixed" else 30000),
                "precision": precision, "h": h}
    if kind == "soft":
        return {"kind": kind, "ic": rng.choice(["sphere", "cloud"]),
                "n": _log_int(rng, 1000, 60000 if precision == "mixed" else 30000),
                "precision": precision, "pot": pot, "h": 0.06}
    if kind == "tree":
        return {"kind": kind, "ic": ic, "n": _log_int(rng, 2000, 400000), "precision": precision,
                "pot": pot, "h": h, "leaf": rng.choice([4, 8, 16])}
    if kind == "bookkeep":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 22), "q_f": rng.choice([0.125, 0.5, 1.0])}
    return {"kind": kind, "ic": rng.choice(["sphere", "plummer"]), "n": _log_int(rng, 1000, 20000),
            "k_max": rng.choice([3, 4, 5]), "precision": "mixed", "h": 1e-2,
            "q_f": rng.choice([0.125, 0.25, 0.5])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, dtype=F64, device="cuda", generator=g)


def _normal(g, *shape):
    return torch.randn(*shape, dtype=F64, device="cuda", generator=g)


def _directions(g, n):
    cz = 2.0 * _uniform(g, n) - 1.0
    ph = 2.0 * math.pi * _uniform(g, n)
    sz = (1.0 - cz * cz).clamp_min(0.0).sqrt()
    return torch.stack([sz * ph.cos(), sz * ph.sin(), cz], 1)


def _morton(pos):
    """The order of the elements along the Morton curve (consecutive ranges are compact)."""
    lo = pos.amin(0)
    ext = (pos.amax(0) - lo).amax().clamp_min(1e-300)
    q = ((pos - lo) / ext * (2 ** 21 - 1)).floor().to(torch.int64)
    key = torch.zeros(pos.shape[0], dtype=torch.int64, device=pos.device)
    for b in range(21):
        for c in range(3):
            key |= ((q[:, c] >> b) & 1) << (3 * b + 2 - c)
    return torch.sort(key, stable=True).indices


def _cloud_velocities(g, pos, grid=64):
    """A Gaussian random velocity field with P(k) ~ k^-4 on a periodic grid over [-1, 1]^3,
    interpolated to the elements, scaled to virial parameter 2."""
    k = torch.fft.fftfreq(grid, dtype=F64, device="cuda") * grid
    kz = torch.fft.rfftfreq(grid, dtype=F64, device="cuda") * grid
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2
    amp = torch.where(k2 > 0, 1.0 / k2.clamp_min(1.0), torch.zeros_like(k2))
    x = (pos + 1.0) * (0.5 * grid)
    i0 = x.floor().to(torch.int64)
    t = x - i0
    vel = torch.zeros_like(pos)
    for c in range(3):
        noise = torch.complex(_normal(g, *k2.shape), _normal(g, *k2.shape))
        f = torch.fft.irfftn(noise * amp, s=(grid, grid, grid))
        for corner in range(8):
            d = [(corner >> b) & 1 for b in range(3)]
            w = torch.ones_like(t[:, 0])
            for b in range(3):
                w = w * (t[:, b] if d[b] else 1.0 - t[:, b])
            j = [(i0[:, b] + d[b]) % grid for b in range(3)]
            vel[:, c] += w * f[j[0], j[1], j[2]]
    vel -= vel.mean(0)
    return vel * (0.6 / (0.5 * (vel * vel).sum(1).mean())).sqrt()


def _initial(ic, n, g):
    """Positions, velocities and equal masses (total 1), along the Morton curve."""
    if ic == "pancake":
        side = round(n ** (1.0 / 3.0))
        k = (torch.arange(side, dtype=F64, device="cuda") + 0.5) / side
        q = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
        disp = 0.8 / (2.0 * math.pi) * torch.sin(2.0 * math.pi * q[:, 0])
        pos = q.clone()
        pos[:, 0] += disp
        pos = torch.remainder(pos + (_uniform(g, n, 3) - 0.5) * (0.01 / side), 1.0)
        vel = 1e-3 * _normal(g, n, 3)
        vel[:, 0] -= disp
    elif ic == "plummer":
        u = 1e-9 + (0.9962 - 1e-9) * _uniform(g, n)           # radii up to 20
        r = 1.0 / (u ** (-2.0 / 3.0) - 1.0).sqrt()
        pos = r[:, None] * _directions(g, n)
        q = torch.zeros(n, dtype=F64, device="cuda")
        todo = torch.ones(n, dtype=torch.bool, device="cuda")
        for _ in range(60):                                   # rejection from q^2 (1 - q^2)^3.5
            x, y = _uniform(g, n), 0.1 * _uniform(g, n)
            ok = todo & (y < x * x * (1.0 - x * x) ** 3.5)
            q = torch.where(ok, x, q)
            todo = todo & ~ok
        v = q * math.sqrt(2.0) * (1.0 + r * r) ** -0.25
        vel = v[:, None] * _directions(g, n)
    else:
        pos = _uniform(g, n).pow(1.0 / 3.0)[:, None] * _directions(g, n)
        if ic == "sphere":
            vel = math.sqrt(0.2) * _normal(g, n, 3)
        else:
            vel = _cloud_velocities(g, pos)
    p = _morton(pos)
    return pos[p].contiguous(), vel[p].contiguous(), torch.full((n,), 1.0 / n, dtype=F64, device="cuda")


def _outputs(n, pot):
    return {"acc": torch.zeros(n, 3, dtype=F64, device="cuda"),
            "jerk": torch.zeros(n, 3, dtype=F64, device="cuda"),
            "tidal": torch.zeros(n, 6, dtype=F64, device="cuda"),
            "pot": torch.zeros(n, dtype=F64, device="cuda") if pot else None,
            "dt_grav": torch.zeros(n, dtype=F64, device="cuda")}


def _due(n, frac, g):
    """Ascending indices of a random due set of about frac n elements."""
    return torch.nonzero(_uniform(g, n) < frac).flatten().to(torch.int32)


def _due_list(n, idx):
    """idx and its count as the compaction leaves them: n entries and a device word."""
    full = torch.zeros(n, dtype=torch.int32, device="cuda")
    full[: idx.numel()] = idx
    return full, torch.tensor([idx.numel()], dtype=torch.int32, device="cuda")


def _params(case, **kw):
    return grav.params(h=case["h"], eta=ETA, precision=PRECISION[case["precision"]],
                       want_pot=bool(case.get("pot", False)), **kw)


def _sizes(case):
    """Sizes spread evenly over the logarithm of the range, in a scattered order."""
    return [int(case["n_min"] * (case["n_max"] / case["n_min"]) ** ((0.6180339887 * (s + 1)) % 1.0))
            for s in range(case["n_sys"])]


def _batch(case, g):
    """Systems packed back to back, alternately Plummer and uniform spheres; 1-50% due in each."""
    sizes = _sizes(case)
    frac = (0.01 + 0.49 * _uniform(g, len(sizes))).cpu()
    parts, idx, offsets, at = [], [], [], 0
    for s, ns in enumerate(sizes):
        parts.append(_initial("plummer" if s % 2 == 0 else "sphere", ns, g))
        idx.append(_due(ns, max(float(frac[s]), 1.5 / ns), g) + at)
        offsets.append(at)
        at += ns
    pos, vel, mass = (torch.cat([p[c] for p in parts]) for c in range(3))
    return pos, vel, mass, offsets, sizes, torch.cat(idx)


def _bookkeeping(case, g):
    n = case["n"]
    dt_min = DT_MAX * 2.0 ** -K_MAX
    return {"dt_min": dt_min, "bin": torch.randint(0, K_MAX + 1, (n,), device="cuda", generator=g).to(torch.int8),
            "tf": torch.zeros(n, dtype=torch.int64, device="cuda"),
            "dt_grav": dt_min * torch.exp(5.0 * _uniform(g, n)),
            "dt_hydro": dt_min * torch.exp(2.0 * _uniform(g, n)),
            "acc": _normal(g, n, 3), "jerk": _normal(g, n, 3)}


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": dict(case), "ws": grav.Workspace()}
    if kind == "bookkeep":
        n = case["n"]
        s.update(_bookkeeping(case, g))
        s.update(active=torch.zeros(n, dtype=torch.uint8, device="cuda"),
                 due=torch.zeros(n, dtype=torch.uint8, device="cuda"),
                 idx=torch.zeros(n, dtype=torch.int32, device="cuda"),
                 count=torch.zeros(1, dtype=torch.int32, device="cuda"),
                 a_out=torch.zeros(n, 3, dtype=F64, device="cuda"), tick=1)
        return s
    if kind == "batched":
        pos, vel, mass, offsets, sizes, idx = _batch(case, g)
        s.update(pos=pos, vel=vel, mass=mass, out=_outputs(mass.numel(), case["pot"]),
                 systems=grav.systems_table(list(zip(offsets, sizes)), device=pos.device),
                 params=_params(case))
        s["idx"], s["count"] = _due_list(mass.numel(), idx)
        return s
    n = case["n"]
    pos, vel, mass = _initial(case["ic"], n, g)
    if kind == "cycle":
        it = AdaptiveIntegrator(pos, vel, mass, h=case["h"], q_f=case["q_f"], k_max=case["k_max"],
                                dt_max=DT_MAX, eta=ETA, precision=PRECISION[case["precision"]],
                                dt_hydro=torch.full((n,), DT_MAX / 4, dtype=F64, device="cuda"))
        it.start()
        it.capture_cycle()
        s["integrator"] = it
        return s
    s.update(pos=pos, vel=vel, mass=mass)
    if kind == "adjoint":
        s["weight"] = _uniform(g, n)
        s["pos"].requires_grad_(True)
        s["mass"].requires_grad_(True)
        return s
    s["out"] = _outputs(n, case["pot"])
    s["params"] = _params(case, box=1.0 if case["ic"] == "pancake" else 0.0)
    if kind == "forces" and case["frac"] < 1.0:
        s["idx"], s["count"] = _due_list(n, _due(n, case["frac"], g))
    if kind == "soft":
        s.update(guess=_guess(case, g), h=torch.zeros(n, dtype=F64, device="cuda"),
                 zeta=torch.zeros(n, dtype=F64, device="cuda"),
                 omega=torch.zeros(n, dtype=F64, device="cuda"), sp=grav.soft_params(),
                 ws_soft=grav.Workspace())
    if kind == "tree":
        s["tp"] = grav.tree_params(theta=0.5, leaf_size=case["leaf"])
    return s


def _guess(case, g):
    """Guesses of the supports: those of the mean density, off by up to 20%."""
    h0 = (32.0 / case["n"]) ** (1.0 / 3.0)
    return h0 * (0.8 + 0.4 * _uniform(g, case["n"]))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "bookkeep":
        tick = s["tick"]
        s["tick"] = tick + 1
        grav.select_due(tick, K_MAX, s["bin"], s["tf"], s["dt_grav"], case["q_f"], s["dt_min"],
                        s["active"], s["due"])
        grav.compact_active(s["due"], s["idx"], s["count"], workspace=s["ws"])
        grav.predict(s["active"], s["due"], s["acc"], s["jerk"], s["tf"], s["dt_min"], s["a_out"])
        grav.assign_bins(tick, K_MAX, DT_MAX, s["active"], s["dt_grav"], s["dt_hydro"], s["bin"])
        return {k: s[k] for k in ("active", "due", "tf", "count", "idx", "a_out", "bin")}
    if kind == "cycle":
        it = s["integrator"]
        it.replay()
        return {"pos": it.pos, "vel": it.vel, "acc": it.acc, "jerk": it.jerk, "tidal": it.tidal,
                "dt_grav": it.dt_grav, "bins": it.bins, "tf": it.tf, "due": it.n_due_total}
    pos, vel, mass = s["pos"], s["vel"], s["mass"]
    n = mass.numel()
    if kind == "adjoint":
        acc, w = gravity(pos, mass, vel, h=case["h"], precision=PRECISION[case["precision"]])
        loss = (s["weight"] * (acc * acc).sum(1)).sum() + w
        g_pos, g_mass = torch.autograd.grad(loss, [pos, mass])
        return {"acc": acc.detach(), "W": w.detach(), "pos_grad": g_pos, "mass_grad": g_mass}
    o = s["out"]
    args = (n, o["acc"], o["jerk"], o["tidal"], o["pot"], o["dt_grav"])
    if kind == "batched":
        grav.eval_batched(s["params"], s["systems"], pos, vel, mass, s["idx"], s["count"], *args,
                          workspace=s["ws"])
        return dict(o)
    if kind == "tree":
        grav.eval_tree(s["params"], s["tp"], pos, vel, mass, None, None, *args, workspace=s["ws"])
        return dict(o)
    if kind == "soft":
        s["h"].copy_(s["guess"])
        grav.soft_solve(s["sp"], pos, mass, s["h"], s["zeta"], s["omega"], workspace=s["ws_soft"])
        grav.eval_soft(s["params"], pos, vel, mass, s["h"], s["zeta"], None, None, *args,
                       workspace=s["ws"])
        return dict(o, h=s["h"], zeta=s["zeta"], omega=s["omega"])
    grav.eval_active(s["params"], pos, vel, mass, s.get("idx"), s.get("count"), *args,
                     workspace=s["ws"])
    return dict(o)


# ---------------------------------------------------------------------------
# what the path cannot do without
# ---------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    pot = bool(case.get("pot", False))
    if kind == "bookkeep":
        # select: bin, T_f in and out, dt_grav, two flags; compaction: flags in, a few indices out;
        # predictor: a, j in, a out for the active; binning: dt_grav is read already, dt_hydro, bin
        return {"bytes": case["n"] * (1 + 16 + 8 + 2 + 1 + 1 + 0.4 * (72 + 8 + 1)), "flops": 6 * case["n"]}
    if kind == "cycle":
        n, ticks = case["n"], 1 << case["k_max"]
        due = 0.1 * n * ticks
        return {"bytes": ticks * n * 72 + due * 152, "flops": due * n * PAIR_FLOPS}
    if kind == "batched":
        mean = (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        square = (case["n_max"] ** 2 - case["n_min"] ** 2) / (2.0 * math.log(case["n_max"] / case["n_min"]))
        due = 0.255
        return {"bytes": case["n_sys"] * mean * (56 + due * (4 + 104 + 8 * pot)),
                "flops": case["n_sys"] * square * due * (PAIR_FLOPS + POT_FLOPS * pot)}
    n = case["n"]
    if kind == "tree":
        return {"bytes": n * (56 + 104 + 8 * pot),
                "flops": n * 50.0 * math.log2(n) * (PAIR_FLOPS + POT_FLOPS * pot)}
    if kind == "adjoint":
        return {"bytes": n * (56 + 8 + 24 + 32 + 32),
                "flops": n * n * (PAIR_FLOPS + POT_FLOPS + ADJOINT_FLOPS)}
    if kind == "soft":
        # about 45 neighbours, 4 iterations, 40 operations of the density sums each
        return {"bytes": n * (56 + 8 + 24 + 104 + 8 * pot),
                "flops": n * (4 * 45 * 40 + n * (PAIR_FLOPS + POT_FLOPS * pot))}
    due = case["frac"] * n
    return {"bytes": n * 56 + due * (4 + 104 + 8 * pot), "flops": due * n * (PAIR_FLOPS + POT_FLOPS * pot)}


# ---------------------------------------------------------------------------
# the same results from plain FP64 tensor operations
# ---------------------------------------------------------------------------

def _spline(u):
    """h^3 f, h^5 g (g = f'/r) and h phi of the cubic spline at u = r / h < 1."""
    u2 = u * u
    ui = 1.0 / u.clamp_min(1e-30)
    f = torch.where(u < 0.5, 32.0 / 3.0 + u2 * (-38.4 + 32.0 * u),
                    64.0 / 3.0 - 48.0 * u + 38.4 * u2 - 32.0 / 3.0 * u * u2 - ui ** 3 / 15.0)
    g = torch.where(u < 0.5, -76.8 + 96.0 * u, -48.0 * ui + 76.8 - 32.0 * u + 0.2 * ui ** 5)
    p = torch.where(u < 0.5, 2.8 + u2 * (-16.0 / 3.0 + u2 * (9.6 - 6.4 * u)),
                    3.2 - ui / 15.0 + u2 * (-32.0 / 3.0 + u * (16.0 + u * (-9.6 + 32.0 / 15.0 * u))))
    return f, g, p


def _kernels(r, h):
    """f, g and phi at separations r with support h (a number or a tensor of r's shape)."""
    ri = 1.0 / r
    f, g, p = ri ** 3, -3.0 * ri ** 5, ri.clone()
    h = torch.as_tensor(h, dtype=F64, device=r.device).expand_as(r)
    inside = r < h
    if bool(inside.any()):
        hi = h[inside]
        a, b, c = _spline(r[inside] / hi)
        f[inside], g[inside], p[inside] = a / hi ** 3, b / hi ** 5, c / hi
    return f, g, p


def _density_slope(u, h):
    """dW/dr of the spline density kernel at u = r / h (0 outside)."""
    dw = torch.where(u < 0.5, u * (-12.0 + 18.0 * u), -6.0 * (1.0 - u) ** 2)
    return torch.where(u < 1.0, 8.0 / (math.pi * h ** 4) * dw, torch.zeros_like(u))


def _chunks(n_t, n):
    step = max(1, min(n_t, (1 << 25) // max(n, 1)))
    return [slice(k, min(n_t, k + step)) for k in range(0, n_t, step)]


def _separations(pos, rows, box):
    d = [pos[None, :, c] - pos[rows, c][:, None] for c in range(3)]
    if box:
        d = [x - box * torch.round(x / box) for x in d]
    r = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]).sqrt()
    own = rows[:, None] == torch.arange(pos.shape[0], device=pos.device)[None, :]
    r[own] = 1.0
    return d, r, own


def _direct(pos, vel, mass, rows, h, pot, box=0.0, supports=None, zeta=None):
    n = mass.numel()
    out = _outputs(n, pot)
    for part in _chunks(rows.numel(), n):
        k = rows[part].long()
        d, r, own = _separations(pos, k, box)
        if supports is None:
            f, g, p = _kernels(r, h)
        else:
            hi, hj = supports[k][:, None].expand_as(r), supports[None, :].expand_as(r)
            f, g, p = (0.5 * (x + y) for x, y in zip(_kernels(r, hi), _kernels(r, hj)))
        m = mass[None, :].expand_as(r).clone()
        m[own] = 0.0
        mf, mg = m * f, m * g
        fa = mf
        if zeta is not None:
            fa = mf - 0.5 * m * (zeta[k][:, None] * _density_slope(r / hi, hi)
                                 + zeta[None, :] * _density_slope(r / hj, hj)) / r
        v = [vel[None, :, c] - vel[k, c][:, None] for c in range(3)]
        dv = mg * (d[0] * v[0] + d[1] * v[1] + d[2] * v[2])
        t6 = torch.zeros(k.numel(), 6, dtype=F64, device=pos.device)
        tr = mf.sum(1)
        for c in range(3):
            out["acc"][k, c] = (fa * d[c]).sum(1)
            out["jerk"][k, c] = (mf * v[c] + dv * d[c]).sum(1)
            t6[:, c] = -(tr + (mg * d[c] * d[c]).sum(1))
        for e, (a, b) in enumerate(((0, 1), (0, 2), (1, 2))):
            t6[:, 3 + e] = -(mg * d[a] * d[b]).sum(1)
        out["tidal"][k] = t6
        if pot:
            out["pot"][k] = -(m * p).sum(1)
        norm2 = (t6[:, :3] ** 2).sum(1) + 2.0 * (t6[:, 3:] ** 2).sum(1)
        out["dt_grav"][k] = math.sqrt(ETA) * (norm2 / 6.0) ** -0.25
    return out


def _adjoint(case, g):
    n = case["n"]
    pos, vel, mass = _initial(case["ic"], n, g)
    weight = _uniform(g, n)
    rows = torch.arange(n, device="cuda")
    fwd = _direct(pos, vel, mass, rows, case["h"], True)
    acc, t6 = fwd["acc"], fwd["tidal"]
    w = 0.5 * (mass * fwd["pot"]).sum()
    a_bar = 2.0 * weight[:, None] * acc
    t = torch.stack([t6[:, [0, 3, 4]], t6[:, [3, 1, 5]], t6[:, [4, 5, 2]]], 1)
    g_pos = (t * a_bar[:, None, :]).sum(2) - mass[:, None] * acc
    g_mass = fwd["pot"].clone()
    for part in _chunks(n, n):
        k = rows[part]
        d, r, own = _separations(pos, k, 0.0)
        f, gk, _ = _kernels(r, case["h"])
        f[own], gk[own] = 0.0, 0.0
        da = d[0] * a_bar[None, :, 0] + d[1] * a_bar[None, :, 1] + d[2] * a_bar[None, :, 2]
        for c in range(3):
            g_pos[k, c] += mass[k] * (f * a_bar[None, :, c] + gk * d[c] * da).sum(1)
        g_mass[k] -= (f * da).sum(1)
    return {"acc": acc, "W": w, "pos_grad": g_pos, "mass_grad": g_mass}


def _supports(pos, mass, h):
    """Solution of (4 pi / 3) h^3 rho(h) = 32 m with Omega and zeta, by Newton steps limited to a
    factor of 2, then the sums at the solution."""
    n = mass.numel()
    h = h.clone()
    rho, rho_h, psi_h = (torch.zeros(n, dtype=F64, device=pos.device) for _ in range(3))
    rows = torch.arange(n, device=pos.device)
    for part in _chunks(n, n):
        k = rows[part]
        _, r, own = _separations(pos, k, 0.0)
        r[own] = 0.0
        near = torch.nonzero(r < 3.0 * h[k][:, None])
        i, j = near[:, 0], near[:, 1]
        rij, mj, hk = r[i, j], mass[j], h[k].clone()
        other = mj * (j != k[i])
        for step in range(60):
            hh = hk[i]
            u = rij / hh
            wu = torch.where(u < 0.5, 1.0 + u * u * (6.0 * u - 6.0), 2.0 * (1.0 - u).clamp_min(0.0) ** 3)
            du = torch.where(u < 0.5, u * (18.0 * u - 12.0), -6.0 * (1.0 - u).clamp_min(0.0) ** 2)
            c = 8.0 / (math.pi * hh ** 3)
            s = lambda x: torch.zeros_like(hk).index_add_(0, i, x)
            ro, rh = s(mj * c * wu), s(-mj * c / hh * (3.0 * wu + u * du))
            if step == 59:
                dup = torch.where(u < 0.5, 2.8 + u ** 2 * (-16.0 + u ** 2 * (48.0 - 38.4 * u)),
                                  3.2 + u ** 2 * (-32.0 + u * (64.0 + u * (-48.0 + 12.8 * u))))
                ps = s(-other * torch.where(u < 1.0, dup, torch.zeros_like(u)) / hh ** 2)
                break
            vol = 4.0 * math.pi / 3.0 * hk ** 3
            new = hk - (vol * ro - 32.0 * mass[k]) / (4.0 * math.pi * hk ** 2 * ro + vol * rh)
            hk = torch.minimum(torch.maximum(new, 0.5 * hk), 2.0 * hk)
        # (the neighbours within three guesses hold every support that was found)
        assert bool((hk < 3.0 * h[k]).all())
        h[k], rho[k], rho_h[k], psi_h[k] = hk, ro, rh, ps
    omega = 1.0 + h * rho_h / (3.0 * rho)
    return h, -h * psi_h / (3.0 * rho * omega), omega


def exact(case, seed):
    """What run() returns for the first pass, in plain FP64; None for the tree (its result is
    defined by its opening decisions) and for a cycle of ticks."""
    g = _gen(seed)
    kind = case["kind"]
    pot = bool(case.get("pot", False))
    if kind in ("tree", "cycle"):
        return None
    if kind == "bookkeep":
        b = _bookkeeping(case, g)
        step = torch.ones_like(b["tf"]) << (K_MAX - b["bin"].long())
        active = 1 % step == 0
        elapsed = torch.where(active, step, torch.zeros_like(step)) * b["dt_min"]
        due = active & (elapsed >= case["q_f"] * b["dt_grav"])
        a = torch.where(due[:, None], b["acc"], b["acc"] + b["jerk"] * elapsed[:, None])
        out = {k: None for k in ("active", "due", "tf", "count", "idx", "bin")}
        out["a_out"] = torch.where(active[:, None], a, torch.zeros_like(a))
        return out
    if kind == "adjoint":
        return _adjoint(case, g)
    if kind == "batched":
        pos, vel, mass, offsets, sizes, idx = _batch(case, g)
        out = _outputs(mass.numel(), pot)
        for at, ns in zip(offsets, sizes):
            own = slice(at, at + ns)
            rows = idx[(idx >= at) & (idx < at + ns)] - at
            part = _direct(pos[own], vel[own], mass[own], rows, case["h"], pot)
            for k in out:
                if out[k] is not None:
                    out[k][own] = part[k]
        return out
    n = case["n"]
    pos, vel, mass = _initial(case["ic"], n, g)
    rows = torch.arange(n, device="cuda")
    if kind == "soft":
        h, zeta, omega = _supports(pos, mass, _guess(case, g))
        return dict(_direct(pos, vel, mass, rows, case["h"], pot, supports=h, zeta=zeta),
                    h=h, zeta=zeta, omega=omega)
    if case["frac"] < 1.0:
        rows = _due(n, case["frac"], g)
    return _direct(pos, vel, mass, rows, case["h"], pot, box=1.0 if case["ic"] == "pancake" else 0.0)
