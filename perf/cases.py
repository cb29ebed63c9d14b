"""Measured cases of the TSBTS framework, each one call (or the few calls a
program makes together) through the public entry points of
``paper_1205_2288_gb300``:

  force     tsbts_force: forces, potentials and step criteria of an active
            set against all bodies, device tensors in and out
  era       Simulation: set_state (a checkpoint) -> step_era -> state
  ensemble  tsbts_init_ensemble on a kept context -> step_era -> state
  adjoint   the differentiable replay of a block schedule and its gradient
            (paper_1205_2288_gb300.autograd)

Sizes are those of the paper's and this repository's own workloads: Plummer
spheres in standard units (n = 256 in FP64 with a fixed era; n = 16384 with
dynamic eras; n = 131072 for the force sweep and a full-size era), 512
Salpeter clusters of 64 to 4096 bodies, the adjoint at n = 8192 and n = 600,
and the force tests' ragged 20000 / 5000 and 4099 / 129.

Results of the mixed path are kept in 32 bits wherever they are sums of its
32-bit pair terms (accelerations, potentials, criteria, gradients): the
order of those sums follows work plans measured in each process, so 32 bits
is what two runs of one program agree on. Positions, velocities and
everything of the FP64 path are kept in 64 bits, block times and steps as
whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1205_2288_gb300 import autograd, inputs, tsbts

DEV = "cuda:0"
K_MAX = 20               # ticks per time unit: 2^20 (the library's default)
ETA = 0.01
DT_MAX = 1.0 / 8.0
# FMA-pipe operations of one pair term of Eq. 3 (bench.py's count), and of
# one pair of the force's vector-Jacobian product (both sides)
OPS_PAIR = 20
OPS_VJP = 39


def listed():
    return [
        # one body re-evaluated against a full-size system: the lone closest
        # encounter of a block step; latency and one pass over the bodies
        {"name": "force_mixed_131072_act1", "kind": "force",
         "precision": "mixed", "n": 131072, "n_act": 1, "eps": 1 / 512},
        # a middling active set of the same system (the force sweep)
        {"name": "force_mixed_131072_act1024", "kind": "force",
         "precision": "mixed", "n": 131072, "n_act": 1024, "eps": 1 / 512},
        # every body: the start of an integration and its largest block steps
        {"name": "force_mixed_131072_all", "kind": "force",
         "precision": "mixed", "n": 131072, "n_act": 131072, "eps": 1 / 512},
        # ragged sizes of the force tests
        {"name": "force_mixed_20000_act5000", "kind": "force",
         "precision": "mixed", "n": 20000, "n_act": 5000, "eps": 1 / 512},
        # the plain FP64 path the mixed one is compared with
        {"name": "force_fp64_20000_act5000", "kind": "force",
         "precision": "fp64", "n": 20000, "n_act": 5000, "eps": 1 / 512},
        # FP64 with sums in ascending order (the reproducible path of n up
        # to 8192), a small ragged active set
        {"name": "force_fp64_4099_act129", "kind": "force",
         "precision": "fp64", "n": 4099, "n_act": 129, "eps": 0.01},
        # Plummer 256, FP64, fixed era 1/8: one era of the latency-bound,
        # bit-reproducible integration, with its energy check
        {"name": "era_fp64_256", "kind": "era", "precision": "fp64",
         "n": 256, "eps": 0.01, "era": "fixed", "span_log2": 3},
        # Plummer 16384, mixed, dynamic eras: the headline integration
        {"name": "era_mixed_16384", "kind": "era", "precision": "mixed",
         "n": 16384, "eps": 1 / 256, "era": "dynamic", "span_log2": 6},
        # Plummer 131072, mixed: the beginning of a full-size era
        {"name": "era_mixed_131072", "kind": "era", "precision": "mixed",
         "n": 131072, "eps": 1 / 512, "era": "fixed", "span_log2": 10},
        # 512 Salpeter clusters of 64..4096 bodies integrated together
        {"name": "ensemble_mixed_512", "kind": "ensemble",
         "precision": "mixed", "clusters": 512, "size": 0, "span_log2": 6},
        # loss and gradient through a pass of block steps at n = 8192
        {"name": "adjoint_mixed_8192", "kind": "adjoint",
         "precision": "mixed", "n": 8192, "eps": 0.01, "passes": 1,
         "span_log2": 5},
        # replay and vector-Jacobian product through all three passes, FP64
        {"name": "adjoint_fp64_600", "kind": "adjoint", "precision": "fp64",
         "n": 600, "eps": 0.01, "passes": 3, "span_log2": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["force"] * 4 + ["era"] * 3 + ["ensemble"] +
                      ["adjoint"] * 2)
    eps = rng.choice([1 / 512, 1 / 256, 0.01])
    if kind == "force":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        n = _log_int(rng, 64, 131072 if precision == "mixed" else 24000)
        n_act = _log_int(rng, 1, n if precision == "mixed" else
                         min(n, 5000))
        return {"kind": kind, "precision": precision, "n": n, "n_act": n_act,
                "eps": eps}
    if kind == "era":
        precision = rng.choice(["mixed", "mixed", "fp64"])
        n = _log_int(rng, 100, 60000 if precision == "mixed" else 1000)
        span = 4 if precision == "fp64" else (6 if n <= 16384 else 9)
        return {"kind": kind, "precision": precision, "n": n, "eps": eps,
                "era": rng.choice(["fixed", "dynamic"]), "span_log2": span}
    if kind == "ensemble":
        if rng.random() < 0.5:
            return {"kind": kind, "precision": "mixed",
                    "clusters": _log_int(rng, 16, 400), "size": 0,
                    "span_log2": 6}
        # equal models integrated together, as in the paper's Sec. 4 study
        return {"kind": kind, "precision": "fp64",
                "clusters": _log_int(rng, 4, 16),
                "size": _log_int(rng, 64, 400), "span_log2": 4}
    precision = rng.choice(["mixed", "fp64"])
    n = _log_int(rng, 300, 8192 if precision == "mixed" else 1000)
    return {"kind": kind, "precision": precision, "n": n, "eps": 0.01,
            "passes": rng.choice([1, 3]) if n <= 1000 else 1,
            "span_log2": 5}


def _precision(case):
    return tsbts.TSBTS_MIXED if case["precision"] == "mixed" else \
        tsbts.TSBTS_FP64


def _span_ticks(case):
    return 1 << (K_MAX - case["span_log2"])


# ---------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------
def _ensemble_inputs(case, seed):
    nc, models = case["clusters"], []
    # sizes: those of the seed-0 ensemble, or all equal
    sizes = np.full(nc, case["size"], np.int64) if case["size"] else \
        inputs.ensemble_sizes(nc, 0)
    for c, n in enumerate(int(x) for x in sizes):
        masses = None if case["size"] else \
            inputs.salpeter_masses(n, 15485863 * (seed + 1) + 2 * c)
        models.append(inputs.plummer(n, 15485863 * (seed + 1) + 2 * c + 1,
                                     masses))
    off = np.zeros(nc + 1, np.int64)
    off[1:] = np.cumsum(sizes)
    return (off, *(np.concatenate([x[k] for x in models]) for k in range(3)),
            np.full(nc, 0.01) if case["size"] else 4.0 / sizes)


def _schedule(m, r, v, eps, span):
    """A pass of block steps over `span` ticks: body i takes the largest
    power-of-two step below eta / sqrt(q_i) of the start (Eq. 3, Eq. 4) and
    is active at its multiples. (step_tau, step_off, act)."""
    m, r, v = (torch.from_numpy(x).to(DEV) for x in (m, r, v))
    n = m.shape[0]
    q = torch.empty(n, dtype=torch.float64, device=DEV)
    for i0 in range(0, n, 1024):
        i1 = min(n, i0 + 1024)
        s2 = ((r[None] - r[i0:i1, None]) ** 2).sum(-1) + eps * eps
        w2 = ((v[None] - v[i0:i1, None]) ** 2).sum(-1)
        c = torch.maximum(w2 / s2, m[None] / (s2 * s2.sqrt()))
        c[torch.arange(i1 - i0), torch.arange(i0, i1)] = 0.0
        q[i0:i1] = c.amax(1)
    dt = (ETA / q.sqrt()).cpu().numpy()
    e = np.frexp(dt)[1] - 1                       # 2^e <= dt < 2^(e + 1)
    step = 1 << np.clip(e + K_MAX, 0, int(math.log2(span))).astype(np.int64)
    tau = np.arange(1, span // int(step.min()) + 1) * int(step.min())
    low = np.minimum(tau & -tau, span)            # who is active: step | tau
    active = {int(b): np.flatnonzero(step <= b).astype(np.int32)
              for b in np.unique(low)}
    parts = [active[int(b)] for b in low]
    off = np.zeros(len(parts) + 1, np.int64)
    np.cumsum([len(p) for p in parts], out=off[1:])
    return tau, off, np.concatenate(parts)


def _cotangents(n, seed):
    g = inputs.rng(seed + 77)
    return g.standard_normal((n, 3)), g.standard_normal((n, 3))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        off, m, r, v, eps = _ensemble_inputs(case, seed)
        ens = tsbts.Ensemble(off, m, r, v, eps=eps, eta=ETA, dt_max=DT_MAX,
                             precision=_precision(case), era_log2=3,
                             k_max=K_MAX)
        return {"case": case, "ens": ens, "in": (off, m, r, v, eps)}
    n = case["n"]
    m, r, v = inputs.plummer(n, seed)
    if kind == "force":
        idx = inputs.active_subset(n, case["n_act"], seed + 1)
        na = case["n_act"]
        s = {"case": case}
        for k, x in dict(m=m, r=r, v=v, idx=idx).items():
            s[k] = torch.from_numpy(x).to(DEV)
        s["out"] = torch.empty(5 * na, dtype=torch.float64, device=DEV)
        s["a"] = s["out"][:3 * na].view(na, 3)
        s["phi"] = s["out"][3 * na:4 * na]
        s["q"] = s["out"][4 * na:]
        return s
    if kind == "era":
        sim = tsbts.Simulation(
            m, r, v, eps=case["eps"], eta=ETA, dt_max=DT_MAX,
            precision=_precision(case), n_iter=3,
            era_mode=1 if case["era"] == "dynamic" else 0, era_log2=3,
            k_max=K_MAX)
        return {"case": case, "sim": sim, "start": sim.checkpoint()}
    sched = _schedule(m, r, v, case["eps"], _span_ticks(case))
    kw = {"passes": [sched] * 3} if case["passes"] == 3 else \
        {"schedule": sched}
    adj = autograd.make_adjoint(n, case["eps"], precision=_precision(case),
                                k_max=K_MAX, **kw)
    s = {"case": case, "adj": adj}
    for k, x in dict(m=m, r=r, v=v).items():
        s[k] = torch.from_numpy(x).to(DEV).requires_grad_()
    s["gr"], s["gv"] = (torch.from_numpy(x).to(DEV)
                        for x in _cotangents(n, seed))
    return s


# ---------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind, mixed = case["kind"], case["precision"] == "mixed"
    if kind == "force":
        tsbts.tsbts_force(_precision(case), s["m"], s["r"], s["v"],
                          case["eps"], s["idx"], s["a"], s["phi"], s["q"])
        if not mixed:
            return {"a": s["a"], "phi": s["phi"], "q": s["q"]}
        na, out = case["n_act"], s["out"].float()
        return {"a": out[:3 * na].view(na, 3), "phi": out[3 * na:4 * na],
                "q": out[4 * na:]}
    if kind == "adjoint":
        x = (s["r"], s["v"], s["m"])
        if mixed:
            loss = autograd.era_loss(s["adj"], *x)
            g = torch.autograd.grad(loss, x)
            return {"loss": loss.detach().float(), "g_r": g[0].float(),
                    "g_v": g[1].float(), "g_m": g[2].float()}
        rT, vT = autograd.replay(s["adj"], *x)
        g = torch.autograd.grad((rT, vT), x, (s["gr"], s["gv"]))
        return {"r": rT.detach(), "v": vT.detach(), "g_r": g[0], "g_v": g[1],
                "g_m": g[2]}
    t_end = 2.0 ** -case["span_log2"]
    if kind == "era":
        sim = s["sim"]
        sim.set_state(s["start"])
    else:
        sim = s["ens"]
        off, m, r, v, eps = s["in"]
        tsbts.tsbts_init_ensemble(sim.ctx, off, m, r, v, eps, ETA, DT_MAX)
    sim.step_era(t_end)
    st = sim.state()
    out = {"r": st["r"], "v": st["v"], "tau": st["tau"], "dt": st["dt"],
           "a": st["a"].astype(np.float32) if mixed else st["a"]}
    if kind == "era" and not mixed:
        out["energy"] = list(sim.energy())
    return out


# ---------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------
def _steps_per_body(n):
    """Steps a body takes per time unit in three passes at eta = 0.01, as
    integrations of 256, 16384 and 131072 bodies took them."""
    return 12600.0 * (n / 16384.0) ** (1.0 / 3.0)


def work(case):
    """bytes: inputs and outputs once; flops: FMA-pipe operations of the
    pair terms (one fused multiply-add counts once)."""
    kind = case["kind"]
    span = 2.0 ** -case.get("span_log2", 0)
    if kind == "force":
        n, na = case["n"], case["n_act"]
        return {"bytes": 56 * n + 44 * na, "flops": OPS_PAIR * n * na}
    if kind == "era":
        n = case["n"]
        pairs = n * n * _steps_per_body(n) * span
        return {"bytes": 200 * n, "flops": OPS_PAIR * pairs}
    if kind == "ensemble":
        # log-uniform sizes in [64, 4096]: mean of N^2 and of N
        ln = math.log(64.0)
        size = case["size"]
        n1 = size or (4096 - 64) / ln
        n2 = size * size or (4096 ** 2 - 64 ** 2) / (2 * ln)
        pairs = case["clusters"] * n2 * _steps_per_body(size or 2000) * span
        return {"bytes": 200 * n1 * case["clusters"],
                "flops": OPS_PAIR * pairs}
    n = case["n"]
    pairs = n * n * _steps_per_body(n) / 3 * span * case["passes"]
    return {"bytes": 112 * n, "flops": (OPS_PAIR + OPS_VJP) * pairs}


# ---------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------
def _exact_force(case, seed):
    m, r, v = (torch.from_numpy(x).to(DEV)
               for x in inputs.plummer(case["n"], seed))
    idx = torch.from_numpy(
        inputs.active_subset(case["n"], case["n_act"], seed + 1)).to(DEV)
    n, na, eps2 = case["n"], case["n_act"], case["eps"] ** 2
    a = torch.empty(na, 3, dtype=torch.float64, device=DEV)
    phi, q = torch.empty_like(a[:, 0]), torch.empty_like(a[:, 0])
    rows = max(1, (1 << 28) // n)
    for k0 in range(0, na, rows):
        i = idx[k0:k0 + rows].long()
        k1 = k0 + i.shape[0]
        at = (torch.arange(k1 - k0, device=DEV), i)
        d = [r[None, :, c] - r[i, None, c] for c in range(3)]
        s2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + eps2
        s = s2.sqrt()
        f = m[None] / (s2 * s)
        f[at] = 0.0
        for c in range(3):
            a[k0:k1, c] = (f * d[c]).sum(1)
        p = m[None] / s
        p[at] = 0.0
        phi[k0:k1] = -p.sum(1)
        w = [v[None, :, c] - v[i, None, c] for c in range(3)]
        w2 = (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]) / s2
        w2[at] = 0.0
        q[k0:k1] = torch.maximum(w2, f).amax(1)
    return {"a": a, "phi": phi, "q": q}


def _force64(p, m, act, eps2):
    d = p[None] - p[act][:, None]
    s2 = (d * d).sum(-1) + eps2
    return ((m[None] / (s2 * s2.sqrt()))[:, :, None] * d).sum(1)


def _exact_replay(case, sched, r0, v0, m):
    """The replay of the schedule's passes with autograd through it: Eq. 2
    (or, in later passes, the cubic Hermite between the previous pass's
    records) places every body, Eq. 1 advances the active ones."""
    eps2 = case["eps"] ** 2
    tau, off, act_all = sched
    n = case["n"]

    def force(p, act):
        if act.shape[0] * n > 1 << 18:
            return checkpoint(_force64, p, m, act, eps2, use_reentrant=False)
        return _force64(p, m, act, eps2)

    a0 = force(r0, torch.arange(n, device=DEV))
    # records of a pass: index j < n is body j's start, n + e its entry e
    nxt = np.full(n + len(act_all), -1, np.int64)
    last = np.arange(n)
    for s in range(len(tau)):
        e = np.arange(off[s], off[s + 1])
        nxt[last[act_all[e]]] = n + e
        last[act_all[e]] = n + e
    nxt = torch.from_numpy(nxt).to(DEV)
    prev = None
    for p in range(case["passes"]):
        r, v, a = r0, v0, a0
        t = torch.zeros(n, dtype=torch.float64, device=DEV)
        recs_r, recs_v = [r0], [v0]
        cur = torch.arange(n, device=DEV)
        for s in range(len(tau)):
            act = torch.from_numpy(act_all[off[s]:off[s + 1]]).to(DEV).long()
            T = float(tau[s]) * 2.0 ** -K_MAX
            h = (T - t)[:, None]
            x = r + v * h + 0.5 * a * h * h
            if prev is not None:
                R, V, tr = prev
                ia, ib = cur, nxt[cur].clamp_min(0)
                H = (tr[ib] - tr[ia])[:, None]
                H = torch.where(H > 0, H, torch.ones_like(H))
                u = (T - tr[ia])[:, None] / H
                w = 1.0 - u
                y = ((1 + 2 * u) * w * w * R[ia] + u * w * w * H * V[ia] +
                     u * u * (3 - 2 * u) * R[ib] -
                     u * u * w * H * V[ib])
                mine = torch.zeros(n, dtype=torch.bool, device=DEV)
                mine[act] = True
                x = torch.where((mine | (nxt[cur] < 0))[:, None], x, y)
            f = force(x, act)
            v = v.index_copy(0, act, v[act] + 0.5 * (a[act] + f) * h[act])
            r = r.index_copy(0, act, x[act])
            a = a.index_copy(0, act, f)
            t = t.clone()
            t[act] = T
            cur = cur.clone()
            cur[act] = n + torch.arange(off[s], off[s + 1], device=DEV)
            recs_r.append(r[act])
            recs_v.append(v[act])
        tr = np.concatenate([np.zeros(n)] + [
            np.full(off[s + 1] - off[s], float(tau[s]) * 2.0 ** -K_MAX)
            for s in range(len(tau))])
        prev = (torch.cat(recs_r), torch.cat(recs_v),
                torch.from_numpy(tr).to(DEV))
    return r, v


def _exact_adjoint(case, seed):
    m, r, v = inputs.plummer(case["n"], seed)
    sched = _schedule(m, r, v, case["eps"], _span_ticks(case))
    x = tuple(torch.from_numpy(y).to(DEV).requires_grad_() for y in (r, v, m))
    rT, vT = _exact_replay(case, sched, *x)
    if case["precision"] == "mixed":
        loss = (x[2] * (rT * rT).sum(1)).sum() / x[2].sum()
        g = torch.autograd.grad(loss, x)
        return {"loss": loss.detach(), "g_r": g[0], "g_v": g[1], "g_m": g[2]}
    gr, gv = (torch.from_numpy(y).to(DEV)
              for y in _cotangents(case["n"], seed))
    g = torch.autograd.grad((rT, vT), x, (gr, gv))
    return {"r": rT.detach(), "v": vT.detach(), "g_r": g[0], "g_v": g[1],
            "g_m": g[2]}


def exact(case, seed):
    """None for integrations: their values are those of the scheme's own
    block steps, which plain torch would take minutes to walk through."""
    if case["kind"] == "force":
        return _exact_force(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    return None
