"""The measured cases: the work a user of this package has it do, through its
public entry points (paper_2304_02731_gb300.qcams and .learned).

A case is a dict of plain values; `kind` says which entry points a pass calls:

  run       init_states -> run_batch -> reduce_xsec of a whole study
  analyze   analyze alone (products of given final states)
  reduce    reduce_xsec alone, with the cross sections read back
  levels    levels of one system (host in, host out)
  train     learned.train of a new network on labelled lanes
  proposal  build_proposal and sample_proposal

Sizes are those of the workload generators, the benchmark's defaults and the
tests, with odd ones among the drawn cases.  The FP64 studies are taken at
sizes a pass of which stays below two seconds.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2304_02731_gb300 import learned as L
from paper_2304_02731_gb300 import qcams as Q
from paper_2304_02731_gb300 import workloads as W

DEV = "cuda"
AMU = 1822.888486209
V_COUNT, J_COUNT = 11, 21          # v in 0..10, j in 0..20: the mixed study's states
SYSTEMS = dict(morse=W.SYS_H2_CA_MORSE, buck=W.SYS_H2_CA_BUCK, lj12=W.SYS_H2_CA_LJ12,
               lj8=W.SYS_H2_CA_LJ8)
MIXED = ["buck", "lj12", "lj8"]
DIMS = {"small": (8, 6, 6, 6, 3), "default": (16, 8, 8, 8, 4), "fine": (32, 16, 16, 8, 5)}


def listed():
    return [
        # the plain study as the README runs it: 1,000 lanes at one energy, six
        # lanes per trajectory; a pass lasts as long as its longest trajectory
        dict(name="plain_1000_hex", kind="run", study="plain", per_b=200, E=0.10, precision=64,
             mode=3),
        # the H2 + Ca sweep (16 energies x 24 impact parameters) in FP64, persistent
        # launch: the method's main path, a first look at 32 lanes per cell, whose
        # low energies hold the longest trajectories
        dict(name="sweep_12288_fp64", kind="run", study="sweep", first=0, per_cell=32,
             precision=64, mode=1),
        # the sweep's upper six energies at 1,536 lanes per cell: full warps
        # throughout, the sweep's throughput
        dict(name="sweep_high_221184_fp64", kind="run", study="sweep", first=10, per_cell=1536,
             precision=64, mode=1),
        # the mixed-potential study (Buckingham and two Lennard-Jones forms,
        # random v and j), persistent launch
        dict(name="mixed_200000_fp64", kind="run", study="mixed", n=200_000, precision=64,
             mode=1),
        # the sweep at full size with the FP32 integrator
        dict(name="sweep_3145728_fp32", kind="run", study="sweep", first=0, per_cell=8192,
             precision=32, mode=1),
        # labelled lanes for the learned proposal: 1 M lanes of LJ(12,6), FP32
        dict(name="train_data_1000000_fp32", kind="run", study="labels", n=1_000_000,
             precision=32, mode=1),
        # products of a million finished lanes of the mixed potentials
        dict(name="analyze_1000000", kind="analyze", n=1_000_000, system="mixed"),
        # products of one plain study: a small call, where launches count
        dict(name="analyze_1000_morse", kind="analyze", n=1000, system="morse"),
        # histograms and cross sections of the mixed study's 2 M lanes
        dict(name="reduce_mixed_2000000", kind="reduce", study="mixed", n=2_000_000,
             weighted=False),
        # the level table of one molecule (a scan over potentials solves it anew each time)
        dict(name="levels_231", kind="levels", n_v=11, n_j=21),
        # one epoch of the outcome network at the benchmark's minibatch
        dict(name="train_1000000x8192", kind="train", n=1_000_000, batch=8192, epochs=1),
        # the default proposal grid and one estimate's 200,000 draws
        dict(name="proposal_200000", kind="proposal", grid="default", n=200_000),
    ]


def _log(rng: random.Random, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["run", "run", "run", "analyze", "reduce", "levels", "train", "proposal"])
    if kind == "run":
        study = rng.choice(["plain", "sweep", "mixed", "labels"])
        precision = 32 if study == "labels" else rng.choice([64, 64, 32])
        if study == "plain":
            return dict(kind=kind, study=study, per_b=_log(rng, 3, 600),
                        E=round(rng.uniform(0.08, 0.30), 3), precision=precision,
                        mode=rng.choice([0, 1] if precision == 32 else [0, 1, 2, 3]))
        mode = rng.choice([1, 1, 0])
        if study == "sweep":
            first = rng.choice([0, rng.randint(8, 15)])
            most = 8192 if precision == 32 else 32 if first == 0 else 1536
            return dict(kind=kind, study=study, first=first, precision=precision, mode=mode,
                        per_cell=_log(rng, 3, most))
        return dict(kind=kind, study=study, precision=precision, mode=mode,
                    n=_log(rng, 301, 200_000 if precision == 64 else 1_000_000))
    if kind == "analyze":
        return dict(kind=kind, n=_log(rng, 100, 1_000_000),
                    system=rng.choice(["mixed", "morse", "lj12"]))
    if kind == "reduce":
        study = rng.choice(["mixed", "sweep"])
        size = dict(n=_log(rng, 1000, 2_000_000)) if study == "mixed" else dict(
            first=0, per_cell=_log(rng, 2, 8192))
        return dict(kind=kind, study=study, weighted=rng.random() < 0.4, **size)
    if kind == "levels":
        return dict(kind=kind, n_v=rng.randint(1, 11), n_j=rng.randint(1, 21))
    if kind == "train":
        batch = _log(rng, 500, 9000)
        return dict(kind=kind, n=batch * rng.randint(2, 120) + rng.randint(0, batch - 1),
                    batch=batch, epochs=1)
    return dict(kind=kind, grid=rng.choice(sorted(DIMS)), n=_log(rng, 1000, 400_000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _workload(case, seed):
    if case["study"] == "plain":
        return W.plain_h2_ca(per_b=case["per_b"], E=case["E"], seed=seed)
    if case["study"] == "sweep":
        wl = W.sweep_h2_ca(per_cell=case["per_cell"], seed=seed)
        return wl.slice(case["first"] * 24 * case["per_cell"], wl.n)   # energies first..15
    if case["study"] == "mixed":
        return W.mixed_ca_h(n=case["n"], seed=seed)
    # labelled lanes of one system: the mixed recipe, LJ(12,6), one cell
    E, b, v, j = L.draw_training_lanes(case["n"], seed)
    n = case["n"]
    return W.Workload("labels", [W.SYS_H2_CA_LJ12], E, b, v, j, np.zeros(n, np.int32),
                      np.zeros(n, np.int32), np.ones(1), np.full(1, L.B2_MAX / 2.0),
                      np.zeros(1, np.int32), 1, seed=seed)


def _on_device(wl):
    f = lambda a, t: torch.as_tensor(np.ascontiguousarray(a), dtype=t).to(DEV)  # noqa: E731
    return (f(wl.E, torch.float64), f(wl.b, torch.float64), f(wl.v, torch.int32),
            f(wl.j, torch.int32))


def _morse(seed):
    """H2-like Morse molecule of the seed: De, re, alpha within 10 % of H-H's."""
    g = np.random.default_rng(seed)
    _, de, re, al = W.HH_MORSE
    return tuple(float(x * g.uniform(0.95, 1.1)) for x in (de, re, al))


def _params(spec):
    """(kind, parameters) of a pair spec, an lj_fit pair as (m, n, Cm, Cn)."""
    if spec[0] == "lj_fit":
        _, m, n, de, re = spec
        return "lj", (m, n, de * n * re ** m / (m - n), de * m * re ** n / (m - n))
    return spec[0], tuple(spec[1:])


def _pot(pair, r, order=0):
    """V (order 0) or V' (order 1) of a pair at r, plain FP64 formulas."""
    kind, p = pair
    if kind == "morse":
        x = torch.exp(-p[2] * (r - p[1]))
        return p[0] * (1 - x) ** 2 - p[0] if order == 0 else 2 * p[0] * p[2] * x * (1 - x)
    if kind == "lj":
        m, n, cm, cn = p
        if order == 0:
            return cm * r ** -m - cn * r ** -n
        return n * cn * r ** (-n - 1) - m * cm * r ** (-m - 1)
    A, B, c6 = p[:3]
    e = A * torch.exp(-B * r)
    return e - c6 * r ** -6.0 if order == 0 else 6 * c6 * r ** -7.0 - B * e


def _masses(spec):
    a, b, c = (m * AMU for m in spec["mass_u"])
    return a, b, c, a * b / (a + b), c * (a + b) / (a + b + c)


def _jacobi_pairs(spec, q1, q2):
    """AB, BC and CA vectors from the Jacobi vectors (also of velocities)."""
    a, b, *_ = _masses(spec)
    return q1, q2 - a / (a + b) * q1, q2 + b / (a + b) * q1


def _hamiltonian(spec, y):
    *_, mu12, mu123 = _masses(spec)
    pairs = [_params(p) for p in spec["pairs"]]
    h = (y[6:9] ** 2).sum(0) / (2 * mu12) + (y[9:12] ** 2).sum(0) / (2 * mu123)
    for pair, r in zip(pairs, _jacobi_pairs(spec, y[0:3], y[3:6])):
        h = h + _pot(pair, (r ** 2).sum(0).sqrt())
    return h


def _finished(spec, n, gen):
    """Final states y[12, n] as runs leave them: one pair bound and the third
    atom beyond r_stop (85 %), all atoms apart (10 %), or a complex still
    together at the time limit (5 %)."""
    u = lambda *s: torch.rand(*s, dtype=torch.float64, device=DEV, generator=gen)  # noqa: E731

    def unit():
        v = torch.randn(3, n, dtype=torch.float64, device=DEV, generator=gen)
        return v / (v ** 2).sum(0).sqrt()

    m = list(_masses(spec)[:3])
    mu12, mu123 = _masses(spec)[3:]
    what = u(n)
    which = (u(n) * 3).long()                       # the bound pair: AB, BC or CA
    pos = torch.zeros(3, 3, n, dtype=torch.float64, device=DEV)   # atom, axis, lane
    vel = torch.zeros_like(pos)
    for k, (a, b, c) in enumerate([(0, 1, 2), (1, 2, 0), (2, 0, 1)]):
        sel = which == k
        pair = _params(spec["pairs"][k])
        re = spec["pairs"][k][2] if spec["pairs"][k][0] == "morse" else (
            spec["pairs"][k][4] if spec["pairs"][k][0] == "lj_fit" else 8.0)
        mu = m[a] * m[b] / (m[a] + m[b])
        r = re * (0.92 + 0.3 * u(n))
        r = torch.where(what > 0.85, torch.where(what > 0.95, r, 12.0 + 20.0 * u(n)), r)
        depth = torch.clamp(-_pot(pair, r), min=1e-5)
        kin = torch.where((what > 0.85) & (what <= 0.95), 0.02 + 0.2 * u(n), depth * 0.9 * u(n))
        dr, dv = unit(), unit()
        far = torch.where(what > 0.95, 3.0 + 2.0 * u(n), 35.0 + 3.0 * u(n))
        out = unit()
        rel = r * dr, (2 * kin / mu).sqrt() * dv
        mab = m[a] + m[b]
        mu3 = m[c] * mab / (mab + m[c])
        jac = far * out, (2 * (0.01 + 0.3 * u(n)) / mu3).sqrt() * out
        for dst, x, X in ((pos, rel[0], jac[0]), (vel, rel[1], jac[1])):
            at = {a: -m[b] / mab * x, b: m[a] / mab * x, c: X}   # x = r_b - r_a
            for atom in range(3):
                dst[atom] = torch.where(sel, at[atom], dst[atom])
    mab = m[0] + m[1]

    def jac12(q):
        return q[1] - q[0], q[2] - (m[0] * q[0] + m[1] * q[1]) / mab

    (r1, r2), (v1, v2) = jac12(pos), jac12(vel)
    status = torch.where(what > 0.95, Q.LANE["DONE_TMAX"], Q.LANE["DONE_RSTOP"]).to(torch.uint8)
    return torch.cat([r1, r2, mu12 * v1, mu123 * v2]), status


def _final_states(case, seed):
    """(system names, sys_id, y, status, E0) of an analyze case."""
    names = MIXED if case["system"] == "mixed" else [case["system"]]
    n = case["n"]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    cut = [n * k // len(names) for k in range(len(names) + 1)]
    parts = [_finished(SYSTEMS[s], hi - lo, gen) for s, lo, hi in zip(names, cut, cut[1:])]
    y = torch.cat([p[0] for p in parts], 1).contiguous()
    status = torch.cat([p[1] for p in parts])
    E0 = torch.cat([_hamiltonian(SYSTEMS[s], y[:, lo:hi]) for s, lo, hi in zip(names, cut, cut[1:])])
    # the energy drift of an integrated lane
    E0 = E0 + 1e-9 * torch.randn(n, dtype=torch.float64, device=DEV, generator=gen)
    sid = torch.cat([torch.full((hi - lo,), k, dtype=torch.int32, device=DEV)
                     for k, (lo, hi) in enumerate(zip(cut, cut[1:]))])
    return names, cut, sid, y, status, E0


def _outcomes(case, seed):
    """Outcome arrays of a reduce case: classes, bins, weights as runs give them."""
    wl = _workload(case, seed)
    n = wl.n
    gen = torch.Generator(device=DEV).manual_seed(seed)
    u = lambda: torch.rand(n, device=DEV, generator=gen, dtype=torch.float64)  # noqa: E731
    edges = torch.tensor([0.62, 0.70, 0.78, 0.93, 0.99], device=DEV, dtype=torch.float64)
    cls = torch.bucketize(u(), edges).to(torch.uint8)
    good = cls <= 2
    vt = torch.where(good, (-3.0 * torch.log1p(-u())).long(), 0).to(torch.int16)
    jt = torch.where(good, (40.0 * u() ** 2).long(), 0).to(torch.int16)
    dv = u() - 0.5
    sg = Q.GB_SIGMA_DEFAULT
    gbw = torch.where(good, torch.exp(-dv ** 2 / (2 * sg * sg)) / (sg * math.sqrt(2 * math.pi)),
                      torch.zeros_like(dv))
    isw = 0.2 + 3.0 * u() if case["weighted"] else None
    return wl, cls, vt, jt, gbw, isw


def _labelled(case, seed):
    """Network inputs x[n, 8] and outcome classes of n lanes."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n = case["n"]
    u = torch.rand(n, 8, device=DEV, generator=gen, dtype=torch.float64)
    x = torch.stack([0.05 + 0.25 * u[:, 0], 10.0 * u[:, 1].sqrt(), (11 * u[:, 2]).floor(),
                     (21 * u[:, 3]).floor(), torch.acos(2 * u[:, 4] - 1), 2 * math.pi * u[:, 5],
                     u[:, 6], 2 * math.pi * u[:, 7]], 1).float().contiguous()
    # reactive at small b and large v, dissociating at high E and v, else quenched
    t = torch.rand(n, device=DEV, generator=gen)
    p_r = 0.6 * torch.exp(-(x[:, 1] / 5.0) ** 2) * (0.3 + 0.07 * x[:, 2])
    p_d = 0.8 * x[:, 0] * x[:, 2] / 10.0
    cls = torch.where(t < p_r, torch.where(t < 0.5 * p_r, 1, 2), torch.where(t < p_r + p_d, 3, 0))
    cls = torch.where(torch.rand(n, device=DEV, generator=gen) < 0.01, 4, cls)
    return x, cls.to(torch.uint8).contiguous()


def _net(seed):
    """Parameters of a trained-looking network (twice the initial scale)."""
    g = np.random.default_rng(seed)
    parts = []
    for n_out, n_in in ((64, 8), (64, 64), (64, 64), (4, 64)):
        parts += [2.0 * g.uniform(-1, 1, n_out * n_in) / math.sqrt(n_in),
                  0.1 * g.standard_normal(n_out)]
    return np.concatenate(parts).astype(np.float32)


NET_MEAN = (0.175, 6.7, 5.0, 10.0, 1.57, 3.14, 0.5, 3.14)
NET_STD = (0.072, 2.36, 3.16, 6.06, 0.68, 1.81, 0.29, 1.81)


def _spec_of(case, seed):
    g = np.random.default_rng(seed + 1)
    return Q.proposal_spec(g.choice([0.05, 0.10, 0.15]), g.integers(0, 11), g.integers(0, 21),
                           dims=DIMS[case["grid"]])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, seed=seed)
    if kind == "run":
        wl = _workload(case, seed)
        s["wl"] = wl
        s["batch"] = Q.Batch.empty(wl.n, DEV, sys_id=wl.sys_id, cell=wl.cell)
        if case["study"] != "plain":      # the plain study passes host arrays, as the README does
            s["in"] = _on_device(wl)
        s["systems"] = Q.systems_array(wl.systems)
        integ = wl.integ if case["precision"] == 64 else W.INTEG_FP32
        s["integ"] = Q.make_integ(**integ, precision=case["precision"], persistent=case["mode"])
    elif kind == "analyze":
        names, _, sid, y, status, E0 = _final_states(case, seed)
        batch = Q.Batch.empty(case["n"], DEV, sys_id=sid)
        batch.y.copy_(y)
        batch.status.copy_(status)
        batch.f64["E0"].copy_(E0)
        s.update(batch=batch, systems=Q.systems_array([SYSTEMS[k] for k in names]),
                 integ=Q.make_integ())
    elif kind == "reduce":
        wl, cls, vt, jt, gbw, isw = _outcomes(case, seed)
        batch = Q.Batch.empty(wl.n, DEV, sys_id=wl.sys_id, cell=wl.cell, isw=isw)
        for dst, src in ((batch.cls, cls), (batch.vt, vt), (batch.jt, jt),
                         (batch.f64["gbw"], gbw)):
            dst.copy_(src)
        s.update(batch=batch, wl=wl)
    elif kind == "levels":
        v, j = np.meshgrid(np.arange(case["n_v"]), np.arange(case["n_j"]), indexing="ij")
        spec = dict(W.SYS_H2_CA_MORSE, pairs=(("morse", *_morse(seed)),) + W.SYS_H2_CA_MORSE["pairs"][1:])
        s.update(systems=Q.systems_array([spec]), v=v.ravel(), j=j.ravel(),
                 sid=np.zeros(v.size, np.int32))
    elif kind == "train":
        s["x"], s["cls"] = _labelled(case, seed)
    else:
        mlp = Q.MLP(DEV, seed=0)
        mlp.set_params(_net(seed))
        mlp.set_standardizer(NET_MEAN, NET_STD)
        s.update(mlp=mlp, spec=_spec_of(case, seed))
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _lanes(batch):
    out = {k: batch.f64[k] for k in ("t", "h", "t_scale", "E0", "dE", "vprime", "jprime", "gbw")}
    out.update({k: getattr(batch, k) for k in ("y", "status", "cls", "nsteps", "nrej", "vt", "jt")})
    return out


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "run":
        wl, batch = s["wl"], s["batch"]
        if case["study"] == "plain":
            _, hist, cells, groups = Q.run_workload(wl, s["integ"], DEV, batch=batch)
            return dict(_lanes(batch), hist=hist, cells=cells, groups=groups)
        Q.init_states(s["systems"], batch, *s["in"], wl.R0, wl.seed, wl.id_offset)
        Q.run_batch(s["systems"], batch, s["integ"])
        if case["study"] == "labels":
            return dict(_lanes(batch), x=Q.mlp_features(batch, *s["in"]))
        hist, cells, groups = Q.reduce_xsec(batch, wl.n_cells, wl.cell_b, wl.cell_w,
                                            wl.cell_group, wl.n_groups)
        return dict(_lanes(batch), hist=hist, cells=cells, groups=groups)
    if kind == "analyze":
        b = s["batch"]
        Q.analyze(s["systems"], b, s["integ"])
        return dict(dE=b.f64["dE"], vprime=b.f64["vprime"], jprime=b.f64["jprime"],
                    gbw=b.f64["gbw"], cls=b.cls, vt=b.vt, jt=b.jt)
    if kind == "reduce":
        wl = s["wl"]
        hist, cells, groups = Q.reduce_xsec(s["batch"], wl.n_cells, wl.cell_b, wl.cell_w,
                                            wl.cell_group, wl.n_groups,
                                            weighted=case["weighted"])
        return dict(hist=hist, cells=cells, groups=groups)
    if kind == "levels":
        lv = Q.levels(s["systems"], s["sid"], s["v"], s["j"])
        return {k: lv[k] for k in ("E", "r_minus", "r_plus", "tau", "ok")}
    if kind == "train":
        mlp = Q.MLP(DEV, seed=s["seed"])
        losses = L.train(mlp, s["x"], s["cls"], epochs=case["epochs"], batch=case["batch"],
                         lr=2e-3, seed=s["seed"])
        return dict(params=mlp.params, m=mlp.m, v=mlp.v, losses=losses)
    q, qfix, cdf = s["mlp"].build_proposal(s["spec"])
    b, u, w, cell = Q.sample_proposal(s["spec"], qfix, cdf, case["n"], s["seed"])
    return dict(q=q, qfix=qfix, cdf=cdf, b=b, u=u, w=w, cell=cell)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# Step attempts per lane of each study (the method's own count at its
# tolerances) and arithmetic operations per attempt, six right-hand sides.
ATTEMPTS = {("plain", 64): 4970, ("sweep", 64): 7610, ("mixed", 64): 2390, ("plain", 32): 990,
            ("sweep", 32): 1520, ("mixed", 32): 470, ("labels", 32): 470}
ATTEMPTS_HIGH = {64: 2710, 32: 540}       # the sweep's upper energies
FLOPS_ATTEMPT = 860.0
LANE_IN = 4 + 4 + 8 + 8 + 4 + 4           # sys_id, cell, E, b, v, j
LANE_STATE = 12 * 8 + 4 * 8 + 1           # y, t_scale, E0, t, h, status
LANE_OUT = 1 + 4 + 4 + 4 * 8 + 2 + 2      # cls, nsteps, nrej, dE, v', j', W, v_t, j_t


def _lanes_of(case):
    if "n" in case:
        return case["n"]
    return 5 * case["per_b"] if case["study"] == "plain" else (
        24 * (16 - case["first"]) * case["per_cell"])


def work(case):
    kind = case["kind"]
    if kind == "run":
        n = _lanes_of(case)
        per_lane = (ATTEMPTS_HIGH[case["precision"]] if case.get("first") else
                    ATTEMPTS[case["study"], case["precision"]])
        return dict(bytes=n * (LANE_IN + LANE_STATE + LANE_OUT), flops=n * per_lane * FLOPS_ATTEMPT)
    if kind == "analyze":
        return dict(bytes=case["n"] * (4 + 1 + 13 * 8 + 37), flops=case["n"] * 1500)
    if kind == "reduce":
        n, cells = _lanes_of(case), 384 if case["study"] == "sweep" else 330
        return dict(bytes=n * (4 + 1 + 2 + 2 + 8 + 8 * case["weighted"]) + cells * Q.H_STRIDE * 16,
                    flops=n * 2)
    if kind == "levels":
        n = case["n_v"] * case["n_j"]
        return dict(bytes=n * 60, flops=n * 8 * 256 * 40)
    if kind == "train":
        steps = case["epochs"] * max(1, case["n"] // case["batch"])
        return dict(bytes=2 * case["n"] * 33 + 4 * 4 * Q.MLP_NPARAMS,
                    flops=steps * case["batch"] * 54e3)
    cells = math.prod(DIMS[case["grid"]])
    return dict(bytes=cells * 24 + case["n"] * (6 * 8 + 4), flops=cells * 18e3 + case["n"] * 100)


# ---------------------------------------------------------------------------
# the same outputs in plain 64-bit torch / numpy
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 words of counters (int64 tensors or numbers) under key = seed."""
    c = [torch.as_tensor(x, dtype=torch.int64, device=DEV) & M32 for x in (c0, c1, c2, c3)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & M32) ^ c[1] ^ k0, b & M32, ((a >> 32) & M32) ^ c[3] ^ k1, a & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _bisect(f, lo, hi, sign, steps=70):
    """Root of f between lo and hi (tensors) where f has `sign` at lo."""
    for _ in range(steps):
        mid = 0.5 * (lo + hi)
        left = f(mid) * sign > 0
        lo, hi = torch.where(left, mid, lo), torch.where(left, hi, mid)
    return 0.5 * (lo + hi)


class _Pair:
    """V_eff of one pair in FP64: barrier, turning points, action and period."""

    def __init__(self, pair, mu):
        self.pair, self.mu = pair, mu
        r = torch.exp(torch.linspace(math.log(0.3), math.log(300.0), 200001, dtype=torch.float64,
                                     device=DEV))
        g = r ** 3 * _pot(pair, r, 1)
        well = torch.argmin(torch.where(r > 0.9, _pot(pair, r), torch.full_like(r, 1e9))) \
            if pair[0] != "buck" else torch.argmin(torch.where(r > 4.5, _pot(pair, r),
                                                               torch.full_like(r, 1e9)))
        one = torch.ones(1, dtype=torch.float64, device=DEV)
        i = int(well)
        self.r_eq = _bisect(lambda x: _pot(pair, x, 1), r[i - 2] * one, r[i + 2] * one, -1.0)
        k = int(torch.argmax(torch.where(r > self.r_eq, g, torch.full_like(g, -1e9))))
        self.r_peak, self.g_max = r[k], float(g[k])
        self.r_b = 0.0
        if pair[0] == "buck":
            d = _pot(pair, r, 1)
            j = int(torch.nonzero((d[:-1] > 0) & (d[1:] <= 0))[0])
            self.r_b = _bisect(lambda x: _pot(pair, x, 1), r[j] * one, r[j + 1] * one, 1.0)
        x, w = np.polynomial.legendre.leggauss(160)
        th = torch.as_tensor(x * math.pi / 2, device=DEV)
        self.sn, self.cs = torch.sin(th), torch.cos(th)
        self.w = torch.as_tensor(w * math.pi / 2, device=DEV)

    def veff(self, r, L2):
        return _pot(self.pair, r) + L2 / (2 * self.mu * r * r)

    def barrier(self, L2):
        """(r_top, threshold, has a well); no barrier within reach: (inf, 0)."""
        c = L2 / self.mu
        f = lambda r: r ** 3 * _pot(self.pair, r, 1) - c  # noqa: E731
        lo = self.r_peak.expand_as(L2).clone()
        hi = lo * 2.0 ** 20
        top = _bisect(f, lo, hi, 1.0, 90)
        none = (L2 <= 0) | (f(hi) >= 0)
        thr = torch.where(none, torch.zeros_like(L2), self.veff(top, L2))
        return torch.where(none, torch.full_like(L2, math.inf), top), thr, (c < self.g_max) | (L2 <= 0)

    def bottom(self, L2):
        c = L2 / self.mu
        return _bisect(lambda r: r ** 3 * _pot(self.pair, r, 1) - c, self.r_eq.expand_as(L2).clone(),
                       self.r_peak.expand_as(L2).clone(), -1.0)

    def action(self, E, L2, r_in, r_top):
        f = lambda r: self.veff(r, L2) - E  # noqa: E731
        lo = self.r_b.expand_as(E).clone() if self.pair[0] == "buck" else r_in / 16.0
        hi = torch.where(torch.isfinite(r_top), r_top, r_in * 4096.0)
        rm, rp = _bisect(f, lo, r_in, 1.0), _bisect(f, r_in, hi, -1.0)
        c, d = 0.5 * (rp + rm), 0.5 * (rp - rm)
        act, per = torch.zeros_like(E), torch.zeros_like(E)
        for s, co, w in zip(self.sn.tolist(), self.cs.tolist(), self.w.tolist()):
            g = torch.clamp(E - self.veff(c + d * s, L2), min=0.0)
            act += w * co * d * g.sqrt()
            per += torch.where(g > 0, w * co * d * g.clamp(min=1e-300).rsqrt(), torch.zeros_like(g))
        return rm, rp, act, per

    def level(self, v, L2):
        s2mu = math.sqrt(2 * self.mu)
        r_top, thr, _ = self.barrier(L2)
        r0 = self.bottom(L2)
        lo = self.veff(r0, L2)
        hi = thr - 1e-10 * (thr - lo)
        exists = s2mu / math.pi * self.action(hi, L2, r0, r_top)[2] - 0.5 >= v
        for _ in range(60):
            E = 0.5 * (lo + hi)
            _, _, act, _ = self.action(E, L2, r0, r_top)
            below = s2mu / math.pi * act - 0.5 < v
            lo, hi = torch.where(below, E, lo), torch.where(below, hi, E)
        E = 0.5 * (lo + hi)
        rm, rp, _, per = self.action(E, L2, r0, r_top)
        return [torch.where(exists, x, torch.zeros_like(x)) for x in (E, rm, rp, s2mu * per)]


def _exact_levels(case, seed):
    a = W.MASS_H2_CA[0] * AMU
    pair = _Pair(("morse", _morse(seed)), a / 2.0)
    v, j = torch.meshgrid(torch.arange(case["n_v"], device=DEV, dtype=torch.float64),
                          torch.arange(case["n_j"], device=DEV, dtype=torch.float64), indexing="ij")
    E, rm, rp, tau = pair.level(v.reshape(-1), (j * (j + 1)).reshape(-1))
    return dict(E=E, r_minus=rm, r_plus=rp, tau=tau, ok=None)


def _exact_analyze(case, seed):
    names, cut, _, y, _, E0 = _final_states(case, seed)
    n = case["n"]
    dE = torch.zeros(n, dtype=torch.float64, device=DEV)
    vp, jp = torch.zeros_like(dE), torch.zeros_like(dE)
    gbw = torch.zeros_like(dE)
    for name, lo, hi in zip(names, cut, cut[1:]):
        spec, ys = SYSTEMS[name], y[:, lo:hi]
        a, b, c, mu12, mu123 = _masses(spec)
        dE[lo:hi] = _hamiltonian(spec, ys) - E0[lo:hi]
        rs = _jacobi_pairs(spec, ys[0:3], ys[3:6])
        vs = _jacobi_pairs(spec, ys[6:9] / mu12, ys[9:12] / mu123)
        mus = (a * b / (a + b), b * c / (b + c), c * a / (c + a))
        found, made = [], []
        for k in range(3):
            p = _Pair(_params(spec["pairs"][k]), mus[k])
            r = (rs[k] ** 2).sum(0).sqrt()
            L2 = mus[k] ** 2 * (torch.linalg.cross(rs[k], vs[k], dim=0) ** 2).sum(0)
            E = 0.5 * mus[k] * (vs[k] ** 2).sum(0) + _pot(p.pair, r)
            r_top, thr, well = p.barrier(L2)
            bound = well & (E < thr) & (r < r_top)
            if p.pair[0] == "buck":
                bound &= (r > p.r_b) & (E < p.veff(p.r_b.expand_as(L2), L2))
            found.append(bound)
            made.append((p, E, L2, r, r_top))
        once = found[0].int() + found[1].int() + found[2].int() == 1
        for bound, (p, E, L2, r, r_top) in zip(found, made):
            i = torch.nonzero(bound & once).reshape(-1)
            if not i.numel():
                continue
            _, _, act, _ = p.action(E[i], L2[i], r[i], r_top[i])
            vp[lo + i] = math.sqrt(2 * p.mu) / math.pi * act - 0.5
            jp[lo + i] = 0.5 * (torch.sqrt(1 + 4 * L2[i]) - 1)
            dv = vp[lo + i] - torch.clamp(torch.floor(vp[lo + i] + 0.5), min=0)
            sg = Q.GB_SIGMA_DEFAULT
            gbw[lo + i] = torch.exp(-dv ** 2 / (2 * sg * sg)) / (sg * math.sqrt(2 * math.pi))
    return dict(dE=dE, vprime=vp, jprime=jp, gbw=gbw, cls=None, vt=None, jt=None)


def _exact_reduce(case, seed):
    if case["weighted"]:
        return None
    wl, cls, *_ = _outcomes(case, seed)
    cell = torch.as_tensor(wl.cell, device=DEV).long()
    cnt = torch.bincount(cell * 6 + cls.long(), minlength=6 * wl.n_cells).view(-1, 6).double()
    N = cnt[:, :5].sum(1, keepdim=True)
    k = torch.cat([cnt, cnt[:, 1:2] + cnt[:, 2:3]], 1)
    P = torch.where(N > 0, k / N.clamp(min=1), torch.zeros_like(k))
    d = torch.where(N > 0, k.sqrt() / N.clamp(min=1) * ((N - k).clamp(min=0) / N.clamp(min=1)).sqrt(),
                    torch.zeros_like(k))
    wb = torch.as_tensor(wl.cell_w * wl.cell_b, device=DEV).view(-1, 1)
    grp = torch.as_tensor(wl.cell_group, device=DEV).long()
    z = torch.zeros(wl.n_groups, 7, dtype=torch.float64, device=DEV)
    sg = 2 * math.pi * z.index_add(0, grp, wb * P)
    se = 2 * math.pi * z.index_add(0, grp, (wb * d) ** 2).sqrt()
    cells, groups = torch.stack([P, d], 2), torch.stack([sg, se], 2)
    return dict(hist=None, cells=cells, groups=groups)


def _forward(params, x):
    at = 0
    for layer, (n_out, n_in) in enumerate(((64, 8), (64, 64), (64, 64), (4, 64))):
        w = params[at:at + n_out * n_in].view(n_out, n_in)
        bias = params[at + n_out * n_in:at + n_out * n_in + n_out]
        at += n_out * n_in + n_out
        x = x @ w.T + bias
        if layer < 3:
            x = x * torch.sigmoid(x)
    return x


def _exact_train(case, seed):
    x, cls = _labelled(case, seed)
    n, batch = case["n"], min(case["batch"], case["n"])
    x = x.double()
    mean, std = x.mean(0), x.std(0, unbiased=False)
    x = (x - mean.float().double()) / std.float().double()
    cls = cls.long()
    p = torch.zeros(Q.MLP_NPARAMS, dtype=torch.float64, device=DEV)
    at = 0
    u = (_philox(torch.arange(Q.MLP_NPARAMS, device=DEV), 0, 3, 0, seed)[0].double() + 0.5) * 2.0 ** -32
    for n_out, n_in in ((64, 8), (64, 64), (64, 64), (4, 64)):
        k = n_out * n_in
        p[at:at + k] = (2 * u[at:at + k] - 1) / math.sqrt(n_in)
        at += k + n_out
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    losses = []
    for step in range(max(1, n // case["batch"])):
        w = _philox(torch.arange(batch, device=DEV), step & M32, step >> 32, 4, seed)
        idx = (w[1] * n + ((w[0] * n) >> 32)) >> 32
        q = p.detach().requires_grad_(True)
        lp = torch.log_softmax(_forward(q, x[idx]), 1)
        c = cls[idx]
        loss = -(lp.gather(1, c.clamp(max=3).view(-1, 1)).view(-1) * (c < 4)).sum() / batch
        g, = torch.autograd.grad(loss, q)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 2e-3 * (m / (1 - 0.9 ** (step + 1))) / ((v / (1 - 0.999 ** (step + 1))).sqrt() + 1e-8)
        losses.append(float(loss))
    return dict(params=p, m=m, v=v, losses=[float(np.mean(losses))])


def _exact_proposal(case, seed):
    g = np.random.default_rng(seed + 1)
    E, v, j = float(g.choice([0.05, 0.10, 0.15])), int(g.integers(0, 11)), int(g.integers(0, 21))
    dims = DIMS[case["grid"]]
    mid = [(torch.arange(d, dtype=torch.float64, device=DEV) + 0.5) / d for d in dims]
    b2, ct, ph, et, ch = (t.reshape(-1) for t in torch.meshgrid(*mid, indexing="ij"))
    one = torch.ones_like(b2)
    x = torch.stack([E * one, (100.0 * b2).sqrt(), v * one, j * one, torch.acos(2 * ct - 1),
                     2 * math.pi * ph, ch, 2 * math.pi * et], 1)
    f64 = dict(dtype=torch.float64, device=DEV)
    x = (x - torch.tensor(NET_MEAN, **f64)) / torch.tensor(NET_STD, **f64)
    pr = torch.softmax(_forward(torch.as_tensor(_net(seed)).to(**f64), x), 1)
    gq = (1e-3 + pr[:, 1] + pr[:, 2]).sqrt()
    q = 0.1 / gq.numel() + 0.9 * gq / gq.sum()
    # the draws invert the integer form of q, rounded network outputs and all: no 64-bit value
    return dict(q=q, qfix=None, cdf=None, b=None, u=None, w=None, cell=None)


def exact(case, seed):
    # the studies' trajectories are chaotic: a 64-bit value of their outputs does not exist
    f = dict(analyze=_exact_analyze, reduce=_exact_reduce, levels=_exact_levels,
             train=_exact_train, proposal=_exact_proposal).get(case["kind"])
    return f(case, seed) if f else None
