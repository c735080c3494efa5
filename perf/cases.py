"""Workloads that stand for what a program does with this library, on one GPU.

``listed()`` names them, ``draw(rng)`` gives another one of the same ranges,
``prepare`` builds what a program holds before the call (context, medium,
geometry, chains that have run for a while, device batches of paths), ``run``
is one pass through the public entry points, ``work`` what that pass cannot do
without and ``exact`` its result in 64 bits where it is a computed number.

Scenes and sizes come from scenes.py, bench.py and the tests: the detector run
the library is benchmarked on, the plain geometry, MALA runs with gradients,
uneven batches of pairs, the layered string of sensors, the paper's two-sensor
scene with tree moves, the optimal bridge, the forward tracer, and the density,
its adjoint and its score on batches of paths.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_1811_04156_gb300 import api
from paper_1811_04156_gb300 import scenes as S

_LAYOUT = {"warp": S.LAYOUT_WARP, "lane": S.LAYOUT_LANE}
_CTX = {}


def listed():
    return [
        # the paper's plain run: few chains, short calls, the estimate and the paths read back each time
        {"name": "plain_small", "kind": "plain", "chains": 64, "steps": 500, "cap": 64, "layout": "warp", "warm": 2000},
        # the benchmark's detector-scale run: every chain stepped, the estimate and the accumulators read
        {"name": "detector", "kind": "detector", "chains": 65536, "steps": 4000, "cap": 256, "layout": "lane",
         "warm": 10000},
        # gradient-informed chains: MALA moves with score accumulation, the gradient read
        {"name": "mala_gradients", "kind": "gradients", "chains": 65536, "steps": 2000, "cap": 64, "layout": "lane",
         "warm": 2000},
        # many pairs at 5-150 m with uneven chain counts and vertex caps of 64-1,024
        {"name": "batched_pairs", "kind": "batched", "pairs": 256, "steps": 1000, "layout": "warp", "warm": 4000},
        # 100 horizontal layers and a string of 60 sensors (general physics, caps of 1,024)
        {"name": "layered_string", "kind": "layered", "sensors": 60, "chains": 512, "steps": 500, "layout": "warp",
         "warm": 3000},
        # one observation interval of the paper's relative-light-yield run: tree moves, then B and the path lengths
        {"name": "two_sensor_tree", "kind": "two_sensor", "chains": 2048, "steps": 200, "b1": 0.3, "cap": 256,
         "warm": 1000},
        # one row of the optimal bridge at the detector geometry: tree moves, reference draws, log ratios
        {"name": "tree_bridge", "kind": "tree_bridge", "chains": 65536, "steps": 200, "draws": 65536, "cap": 256,
         "layout": "lane", "warm": 500},
        # the forward tracer the sampler is compared with
        {"name": "tracer_detector", "kind": "trace", "scene": "detector", "photons": 8_000_000, "cap": 256},
        # the tracer in the two-sensor scene (layers, vMF emission, phase mixture) with path-length histogram
        {"name": "tracer_lengths", "kind": "trace_lengths", "photons": 8_000_000, "cap": 256, "bins": 50, "b1": 0.3},
        # log density of a large batch of a caller's paths
        {"name": "logp_batch", "kind": "logp", "batch": 131072, "cap": 64, "n_hi": 40},
        # density and its gradient with respect to every vertex through autograd, general physics
        {"name": "adjoint_batch", "kind": "adjoint", "batch": 32768, "cap": 128, "n_hi": 96, "b1": 0.3},
        # d log p / d theta of 200 layer parameters per path
        {"name": "score_layers", "kind": "score", "batch": 32768, "cap": 128, "n_hi": 80},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plain", "detector", "gradients", "batched", "layered", "two_sensor", "tree_bridge", "trace",
                       "trace_lengths", "logp", "adjoint", "score"])
    c = {"kind": kind}
    if kind == "plain":
        c.update(chains=_log_int(rng, 16, 2048), steps=_log_int(rng, 100, 4000), cap=rng.randint(17, 64),
                 layout="warp", warm=2000)
    elif kind == "detector":
        c.update(chains=_log_int(rng, 4096, 65536), steps=_log_int(rng, 300, 4000), cap=rng.randint(64, 256),
                 layout="lane", warm=8000)
    elif kind == "gradients":
        c.update(chains=_log_int(rng, 4096, 65536), steps=_log_int(rng, 200, 2000), cap=rng.randint(33, 64),
                 layout="lane", warm=2000)
    elif kind == "batched":
        c.update(pairs=_log_int(rng, 8, 256), steps=_log_int(rng, 100, 1000), layout="warp", warm=4000)
    elif kind == "layered":
        c.update(sensors=rng.randint(3, 60), chains=_log_int(rng, 32, 512), steps=_log_int(rng, 50, 500),
                 layout="warp", warm=2000)
    elif kind == "two_sensor":
        c.update(chains=_log_int(rng, 256, 2048), steps=_log_int(rng, 50, 200), cap=rng.randint(160, 256),
                 b1=rng.choice(S.TWO_SENSOR_B1), warm=600)
    elif kind == "tree_bridge":
        c.update(chains=_log_int(rng, 8192, 65536), steps=_log_int(rng, 20, 200), draws=_log_int(rng, 4096, 65536),
                 cap=rng.randint(96, 256), layout="lane", warm=400)
    elif kind == "trace":
        # bright close sensor: any photon count; at 50 m one photon in 5e5 is detected
        if rng.random() < 0.5:
            c.update(scene="plain", photons=_log_int(rng, 10_000, 8_000_000), cap=rng.randint(24, 64))
        else:
            c.update(scene="detector", photons=_log_int(rng, 3_000_000, 8_000_000), cap=rng.randint(64, 256))
    elif kind == "trace_lengths":
        c.update(photons=_log_int(rng, 3_000_000, 8_000_000), cap=rng.randint(128, 256), bins=rng.randint(20, 200),
                 b1=rng.choice(S.TWO_SENSOR_B1))
    elif kind == "logp":
        cap = rng.randint(16, 128)
        c.update(batch=_log_int(rng, 64, 65536), cap=cap, n_hi=rng.randint(8, cap))
    elif kind == "adjoint":
        cap = rng.randint(24, 256)
        c.update(batch=_log_int(rng, 64, 16384), cap=cap, n_hi=rng.randint(12, cap), b1=rng.choice(S.TWO_SENSOR_B1))
    else:
        cap = rng.randint(24, 256)
        c.update(batch=_log_int(rng, 64, 16384), cap=cap, n_hi=rng.randint(12, cap))
    return c


def _scene(case, seed):
    kind = case["kind"]
    if kind == "plain":
        sc = S.plain(n_chains=case["chains"], n_steps=case["warm"], cap=case["cap"])
    elif kind == "detector":
        sc = S.detector(n_chains=case["chains"], n_steps=case["warm"], cap=case["cap"])
    elif kind == "gradients":
        sc = S.gradients(n_chains=case["chains"], n_steps=case["warm"], cap=case["cap"])
    elif kind == "batched":
        sc = S.batched(n_pairs=case["pairs"], n_steps=case["warm"])
    elif kind == "layered":
        sc = S.layered(n_sensors=case["sensors"], chains_per_sensor=case["chains"], n_steps=case["warm"])
    elif kind == "two_sensor":
        sc = S.two_sensor(case["b1"], n_chains=case["chains"], cap=case["cap"])
        sc.run = dataclasses.replace(sc.run, within=S.WITHIN_TREE, sigma=0.3, burn_in=0)
    elif kind == "tree_bridge":
        # straight starts near the mean vertex count of the equilibrium (15)
        sc = S.detector(n_chains=case["chains"], cap=case["cap"])
        sc.run = dataclasses.replace(sc.run, within=S.WITHIN_TREE, sigma=0.3, burn_in=0, init_k=12)
    elif kind == "trace":
        sc = (S.plain if case["scene"] == "plain" else S.detector)(n_chains=1, cap=case["cap"])
    elif kind in ("trace_lengths", "adjoint"):
        sc = S.two_sensor(case["b1"], n_chains=1, cap=case["cap"])
    elif kind == "logp":
        sc = S.detector(n_chains=1, cap=max(case["cap"], 2))
    else:
        sc = S.layered(n_sensors=60, chains_per_sensor=1, cap=max(case["cap"], 2))
    sc.run = dataclasses.replace(sc.run, seed=S.BASE_SEED + 7919 * seed)
    if "layout" in case:
        sc.run.layout = _LAYOUT[case["layout"]]
    return sc


# pair of the scene that the density cases evaluate (the layered string: a sensor 26 m above the source)
_PAIR = {"logp": 0, "adjoint": 0, "score": 31}


def _paths(sc, pair, batch, cap, n_hi, seed):
    """Paths from the source to points of the sensor that face the last scattering,
    sorted along the line with a lateral spread of a scattering length's order; n in [2, n_hi]."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    p = sc.pairs[pair]
    src = torch.tensor(sc.sources[p.source].pos, dtype=torch.float64, device="cuda")
    cen = torch.tensor(sc.sensors[p.sensor].centre, dtype=torch.float64, device="cuda")
    R = float(sc.sensors[p.sensor].radius)
    n = torch.randint(2, n_hi + 1, (batch,), generator=gen, device="cuda", dtype=torch.int32)
    i = torch.arange(cap, device="cuda")[None, :]
    u = 0.02 + 0.93 * torch.rand(batch, cap, generator=gen, device="cuda", dtype=torch.float64)
    inner = (i >= 1) & (i <= n[:, None] - 2)
    u = torch.where(inner, u, torch.where(i == 0, -1.0, 9.0).to(u.dtype)).sort(dim=1).values
    off = 1.5 * torch.randn(3, batch, cap, generator=gen, device="cuda", dtype=torch.float64)
    x = src[:, None, None] + u * (cen - src)[:, None, None] + off
    x = torch.where(inner, x, torch.where(i == 0, src[:, None, None], torch.zeros_like(x)))
    last = (n.long() - 2)[None, :, None].expand(3, batch, 1)
    nu = x.gather(2, last)[:, :, 0] - cen[:, None]
    nu = nu / nu.norm(dim=0) + 0.3 * torch.randn(3, batch, generator=gen, device="cuda", dtype=torch.float64).clamp(-1.5, 1.5)
    end = cen[:, None] + R * nu / nu.norm(dim=0)
    return torch.where(i == n[:, None] - 1, end[:, :, None], x).float().contiguous(), n


def _context():
    """One context for the process, as a program keeps it (it holds the tuned launch shapes)."""
    if "ctx" not in _CTX:
        _CTX["ctx"] = api.Context(0)
    return _CTX["ctx"]


def prepare(case, seed):
    ctx = _context()
    kind = case["kind"]
    sc = _scene(case, seed)
    st = {"case": case, "ctx": ctx, "scene": sc, "medium": api.Medium(ctx, sc.medium),
          "geom": api.Geometry(ctx, sc.sources, sc.sensors, sc.pairs), "seed": int(seed)}
    if "warm" in case:
        st["chains"] = api.Chains(ctx, st["medium"], st["geom"], sc.run)
        st["chains"].run_steps(case["warm"])
    if kind == "two_sensor":
        st["sums"] = torch.zeros(2 * case["chains"], dtype=torch.float64, device="cuda")
        st["hist"] = torch.zeros((2, 50), dtype=torch.float64, device="cuda")
    if kind in _PAIR:
        st["xyz"], st["n"] = _paths(sc, _PAIR[kind], case["batch"], case["cap"], case["n_hi"], seed)
        if kind == "adjoint":
            st["xyz"].requires_grad_(True)
    torch.cuda.synchronize()
    return st


_EST = ("intensity", "std_err", "pi_direct", "z2", "rhat", "mean_n", "mean_length", "n_samples", "ess")


def _estimates(chains):
    rows = chains.read_estimator()
    return np.array([[r[k] for k in _EST] + list(r["accept"]) + list(r["proposals"]) for r in rows], dtype=np.float64)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    ctx, med, geom = state["ctx"], state["medium"], state["geom"]
    ch = state.get("chains")
    if kind in ("plain", "detector", "batched", "layered", "gradients"):
        ch.run_steps(case["steps"])
        out = {"estimates": _estimates(ch), "accumulators": ch.read_accumulators()}
        if kind == "gradients":
            out["grad"], out["grad_se"] = ch.grad_estimator()
        if kind == "plain":
            out["xyz"], n, steps = ch.read_states()
            out["n"], out["steps"] = n, steps.astype(np.int64)
        return out
    if kind == "two_sensor":
        ch.run_steps(case["steps"])
        row = torch.empty(2 * case["chains"], dtype=torch.float32, device="cuda")
        ch.yield_observe(0, 1, state["sums"])
        ch.yield_observe_log(0, 1, row)
        ch.length_hist(115.0, 215.0, state["hist"])
        return {"sums": state["sums"], "logr": row, "hist": state["hist"]}
    if kind == "tree_bridge":
        ch.run_steps(case["steps"])
        row = torch.empty(case["draws"] + case["chains"], dtype=torch.float32, device="cuda")
        ch.bridge_observe_log(0, case["draws"], 0, 4242 + state["seed"], row)
        return row
    if kind == "trace":
        return api.trace(ctx, med, geom, 0, 99 + state["seed"], case["photons"], max_scatter=case["cap"] - 2)
    if kind == "trace_lengths":
        r, h = api.trace_lengths(ctx, med, geom, 0, 901 + state["seed"], case["photons"], 115.0, 215.0, case["bins"],
                                 r_reject=400.0, max_scatter=case["cap"] - 2)
        return {"result": r, "hist": h}
    if kind == "logp":
        return api.logp(ctx, med, geom, _PAIR[kind], state["xyz"], state["n"])
    if kind == "adjoint":
        lp = api.LogP.apply(state["xyz"], state["n"], (ctx, med, geom, _PAIR[kind]))
        (g,) = torch.autograd.grad(lp, state["xyz"], torch.ones_like(lp))
        return {"logp": lp.detach(), "grad": g}
    return api.score(ctx, med, geom, _PAIR[kind], state["xyz"], state["n"])


def _mean_n(case):
    kind = case["kind"]
    return {"plain": 6, "gradients": 6, "detector": 12, "batched": 70, "layered": 40, "two_sensor": 47,
            "tree_bridge": 15}.get(kind, 0)


def work(case):
    kind = case["kind"]
    if kind in _PAIR:
        b, cap, n = case["batch"], case["cap"], 0.5 * (2 + case["n_hi"])
        read = b * (12 * n + 4)
        if kind == "logp":
            return {"bytes": read + 4 * b, "flops": b * n * 80}
        if kind == "adjoint":
            return {"bytes": read + 4 * b + 12 * b * cap, "flops": b * n * 300}
        return {"bytes": read + 4 * b * 200, "flops": b * n * 40}
    if kind in ("trace", "trace_lengths"):
        # a photon scatters until its limit unless it leaves (r_reject): about 130 operations per flight
        flights = case["cap"] - 1 if kind == "trace" else min(case["cap"] - 1, 130)
        return {"bytes": 400, "flops": case["photons"] * flights * 130.0}
    n = _mean_n(case)
    if kind == "batched":
        total = sum(p.n_chains for p in S.batched(n_pairs=case["pairs"]).pairs)
    elif kind == "layered":
        total = case["sensors"] * case["chains"]
    else:
        total = case["chains"] * (2 if kind == "two_sensor" else 1)
    # random numbers 120; a move of one vertex 90, a birth or death 140 + n (MALA: its two gradients 300 more);
    # a tree move 300 per vertex
    within = 300 * n if kind in ("two_sensor", "tree_bridge") else (390 if kind == "gradients" else 90)
    flops = total * case["steps"] * (120 + 0.6 * within + 0.4 * (140 + n))
    state = total * (2 * 12 * n + 2 * 128 + 24)
    if kind == "two_sensor":
        state += total * (12 * n + 12)
    if kind == "tree_bridge":
        state += total * (12 * n + 4) + 4 * case["draws"]
        flops += (total + case["draws"]) * n * 200
    return {"bytes": state, "flops": flops}


# ---------------------------------------------------------------------------
# 64-bit results of the density cases
# ---------------------------------------------------------------------------
def _unit(v):
    return v / v.norm(dim=0, keepdim=True)


def _tables(med):
    """Layer boundaries (the first and last layer extend to infinity) and coefficients."""
    if med.kind == S.HOMOGENEOUS:
        return [(-math.inf, math.inf, 1.0 / med.lambda_s, 1.0 / med.lambda_a)]
    L = med.n_layers
    return [(-math.inf if l == 0 else med.z0 + l * med.dz, math.inf if l == L - 1 else med.z0 + (l + 1) * med.dz,
             1.0 / float(med.lambda_s_layers[l]), 1.0 / float(med.lambda_a_layers[l])) for l in range(L)]


def _share(zP, zQ, lo, hi):
    """Share of the segment between heights zP and zQ that lies in [lo, hi)."""
    a, b = torch.minimum(zP, zQ), torch.maximum(zP, zQ)
    part = (torch.clamp(b, max=hi) - torch.clamp(a, min=lo)).clamp(min=0.0)
    span = b - a
    flat = ((a >= lo) & (a < hi)).to(a.dtype)
    return torch.where(span > 0, part / torch.where(span > 0, span, torch.ones_like(span)), flat)


def _logp64(sc, pair, x, n):
    med, pr = sc.medium, sc.pairs[pair]
    src, sen = sc.sources[pr.source], sc.sensors[pr.sensor]
    B, cap = x.shape[1], x.shape[2]
    i = torch.arange(cap, device=x.device)[None, :]
    nn = n[:, None].long()
    P, Q = x[:, :, :-1], x[:, :, 1:]
    live = i[:, :-1] <= nn - 2
    far = torch.tensor([1.0, 2.0, 3.0], dtype=x.dtype, device=x.device)[:, None, None]
    r = torch.where(live[None], Q - P, far)
    ell = r.norm(dim=0)
    rh = r / ell
    tab = torch.tensor(_tables(med), dtype=x.dtype, device=x.device)
    b_of, c_of = tab[:, 2], tab[:, 2] + tab[:, 3]
    if med.kind == S.LAYERED:
        # optical depth over the height span from the antiderivative of the coefficient in z
        layer = ((x[2].detach() - med.z0) / med.dz).floor().clamp(0, len(tab) - 1).long()
        floor_z = med.z0 + med.dz * torch.arange(len(tab), dtype=x.dtype, device=x.device)
        F0 = torch.cat([torch.zeros_like(c_of[:1]), (c_of * med.dz).cumsum(0)[:-1]])
        F = F0[layer] + c_of[layer] * (x[2] - floor_z[layer])
        same = layer[:, 1:] == layer[:, :-1]
        span = torch.where(same, torch.ones_like(ell), Q[2] - P[2])
        tau = ell * torch.where(same, c_of[layer[:, 1:]], (F[:, 1:] - F[:, :-1]) / span)
        logb = b_of[layer].log()
    else:
        tau, logb = c_of[0] * ell, b_of[0].log().expand(B, cap)
    seg = -tau - 2.0 * ell.log()
    lp = torch.where(live, seg, torch.zeros_like(seg)).sum(1)
    # scattering vertices
    dm, dp = rh[:, :, :-1] - rh[:, :, 1:], rh[:, :, :-1] + rh[:, :, 1:]
    omc, opc = 0.5 * (dm * dm).sum(0), 0.5 * (dp * dp).sum(0)
    g, f = med.g, med.f_sl
    lhg = math.log(0.5 * (1 - g * g)) - math.log(2 * math.pi) - 1.5 * ((1 - g) ** 2 + 2 * g * omc).log()
    ph = lhg
    if f > 0:
        al = 2 * g / (1 - g)
        lsl = math.log(0.5 * (1 + g) / (1 - g)) - math.log(2 * math.pi) + al * (0.5 * opc).log()
        ph = torch.logaddexp(math.log(1 - f) + lhg, math.log(f) + lsl)
    mid = i[:, 1:-1] <= nn - 2
    lp = lp + torch.where(mid, ph + logb[:, 1:-1], torch.zeros_like(ph)).sum(1)
    # emission
    if src.emission == S.EMIT_VMF:
        d = torch.tensor(src.direction, dtype=x.dtype, device=x.device)
        k = src.kappa
        lp = lp + k * (rh[:, :, 0] * (d / d.norm())[:, None]).sum(0) + math.log(k) - math.log(2 * math.pi) - k \
            - math.log(-math.expm1(-2 * k))
    else:
        lp = lp - math.log(4 * math.pi)
    # detection
    c = torch.tensor(sen.centre, dtype=x.dtype, device=x.device)[:, None]
    last = (nn - 1)[None].expand(3, B, 1)
    nu = _unit(x.gather(2, last)[:, :, 0] - c)
    a_in = rh.gather(2, last - 1)[:, :, 0]
    cphi = -(a_in * nu).sum(0)
    ok = cphi > 0
    lp = lp + torch.where(ok, cphi, torch.ones_like(cphi)).log()
    if sen.rho == S.RHO_PAPER:
        h = torch.tensor(sen.rho_hat, dtype=x.dtype, device=x.device)
        t = (nu * (h / h.norm())[:, None]).sum(0)
        lp = lp + 3 * t - 1 - (2 * t + 0.7).cosh().log()
    # segments that touch the sensor before the last one
    with torch.no_grad():
        w = c[:, :, None] - P
        t = ((w * r).sum(0) / (r * r).sum(0)).clamp(0.0, 1.0)
        hit = ((P + t * r - c[:, :, None]).norm(dim=0) <= sen.radius) & (i[:, :-1] <= nn - 3)
        ok = ok & ~hit.any(1)
    return lp, ok


def exact(case, seed):
    kind = case["kind"]
    if kind not in _PAIR:
        return None
    sc = _scene(case, seed)
    pair = _PAIR[kind]
    xyz, n = _paths(sc, pair, case["batch"], case["cap"], case["n_hi"], seed)
    x = xyz.double()
    minus = torch.tensor(-math.inf, dtype=torch.float64, device="cuda")
    if kind == "logp":
        lp, ok = _logp64(sc, pair, x, n)
        return torch.where(ok, lp, minus)
    if kind == "adjoint":
        x.requires_grad_(True)
        lp, ok = _logp64(sc, pair, x, n)
        (g,) = torch.autograd.grad(torch.where(ok, lp, torch.zeros_like(lp)).sum(), x)
        return {"logp": torch.where(ok, lp, minus).detach(), "grad": g}
    # score: (len_l b_l^2 - n_l b_l, len_l a_l^2) per layer
    i = torch.arange(case["cap"], device="cuda")[None, :]
    nn = n[:, None].long()
    live, inner = i[:, :-1] <= nn - 2, (i >= 1) & (i <= nn - 2)
    ell = torch.where(live, (x[:, :, 1:] - x[:, :, :-1]).norm(dim=0), torch.zeros_like(x[0, :, 1:]))
    tab = _tables(sc.medium)
    out = torch.empty(case["batch"], 2 * len(tab), dtype=torch.float64, device="cuda")
    for l, (lo, hi, b, a) in enumerate(tab):
        length = (ell * _share(x[2, :, :-1], x[2, :, 1:], lo, hi)).sum(1)
        count = (inner & (x[2] >= lo) & (x[2] < hi)).sum(1)
        out[:, l] = length * b * b - count * b
        out[:, len(tab) + l] = length * a * a
    return out
