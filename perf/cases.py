"""Workloads of the decoder that are timed, through its public entry points.

A case is a dict of plain values; `kind` says which entry point it goes through:

  decode    Context.decode: host arrays in, host arrays out, one call per problem
  plan      Plan.run_async + Plan.collect: a problem kept on the device and decoded again
  range     Plan.run_slots_async + Plan.collect: one slot range of a decode that is extended until
            its standard errors are small enough
  batch     Batch.launch_graph + Batch.collect: many uneven instances, one captured graph
  grad      MLP.loss_grad: one training pass of the learned model (forward, loss, backward)
  inputs    learned.features + learned.learned_inputs: scan weights and initial marginals of new
            instances from the trained model

Pooling designs are random k-sets designs with three to six true positives and noisy outcomes, as a
laboratory's library gives them: every clone in `deg` pools (or, mixed, in two to eight), pools of
13 clones' worth of design each unless the case says otherwise.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2608_30239_gb300 import learned, mcpd

DEVICE = "cuda:0"

# Noise settings: the low noise of a clean library, the high noise of a difficult one.
LOW, HIGH = (0.01, 0.05), (0.10, 0.20)


def listed():
    lib = dict(n=1298, m=97, deg=6, pos=3)
    return [
        # The smallest: a tiny problem in one call, every pair run to its meeting once (no refill).
        dict(name="decode_tiny", kind="decode", n=20, m=8, deg=3, pos=2, fp=0.02, fn=0.05, q=0.01, slots=4096,
             horizon=0),
        # The paper's own instance shape: three pools per clone, pruned to 333 clones, a window of
        # three sweeps, a horizon and a meeting cap of 20 sweeps.
        dict(name="plan_pruned_capped", kind="plan", n=1298, m=97, deg=3, pos=3, fp=0.10, fn=0.10, q=2.6 / 1298,
             n_active=333, window_sweeps=3, slots=100000, horizon=6660, cap=6660),
        # The library at low noise: 262,144 slots, a budget of 1e10 site updates.
        dict(name="plan_library", kind="plan", **lib, fp=LOW[0], fn=LOW[1], q=3 / 1298, slots=262144, horizon=19073),
        # The largest: the high-noise library, 524,288 slots, a budget of 4e10 site updates.
        dict(name="plan_high_noise", kind="plan", **lib, fp=HIGH[0], fn=HIGH[1], q=3 / 1298, slots=524288,
             horizon=38146),
        # Learned scan weights and a learned random start.
        dict(name="plan_learned_start", kind="plan", **lib, fp=HIGH[0], fn=HIGH[1], q=3 / 1298, slots=87552,
             horizon=38146, custom=True, init=True),
        # Pairs with a lag of one sweep, the cheapest way to small standard errors here.
        dict(name="plan_lag_sweep", kind="plan", **lib, fp=HIGH[0], fn=HIGH[1], q=3 / 1298, slots=16384,
             horizon=38146, lag=1298),
        # The first range of a decode extended until its errors are small: 1024 slots on a plan
        # shaped for the whole job, so few pairs that the length of one slot sets the time.
        dict(name="range_first", kind="range", **lib, fp=HIGH[0], fn=HIGH[1], q=3 / 1298, slots=524288, range=1024,
             horizon=38146),
        # Clones in two to eight pools, an odd number of clones: the build for any degree.
        dict(name="plan_mixed_degree", kind="plan", n=2003, m=151, deg=0, pos=4, fp=0.05, fn=0.10, q=4 / 2003,
             slots=38912, horizon=20030, cap=40060),
        # Knill's systematic scan, uncoupled: the comparator that every report shows beside it.
        dict(name="plan_systematic", kind="plan", **lib, fp=LOW[0], fn=LOW[1], q=3 / 1298, slots=262144,
             horizon=19073, coupled=False, scan=mcpd.MCPD_SCAN_SYSTEMATIC),
        # Uneven instances (200 to 5000 clones, 4 to 8 pools each) with the paper's meeting cap.
        dict(name="batch_uneven_capped", kind="batch", count=128, n_lo=200, n_hi=5000, slots=512, sweeps=20,
             cap_sweeps=20),
        # One minibatch of training: 64 instances of 1298 clones.
        dict(name="train_grad", kind="grad", count=64, n_lo=1298, n_hi=1298),
        # Learned inputs of 64 new instances, from their designs.
        dict(name="learned_inputs", kind="inputs", count=64, n_lo=1298, n_hi=1298),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode", "plan", "plan", "plan", "plan", "range", "batch", "grad", "inputs"])
    if kind in ("grad", "inputs"):
        lo = _log_int(rng, 50, 2000)
        return dict(kind=kind, count=_log_int(rng, 1, 200), n_lo=lo, n_hi=int(lo * rng.uniform(1.0, 2.5)))
    if kind == "batch":
        lo = _log_int(rng, 100, 1500)
        return dict(kind=kind, count=_log_int(rng, 2, 96), n_lo=lo, n_hi=min(5000, int(lo * rng.uniform(1.0, 8.0))),
                    slots=_log_int(rng, 32, 1024), sweeps=rng.randint(2, 20), cap_sweeps=20)
    n = _log_int(rng, 20, 5000)
    m = max(8, int(round(n / rng.uniform(11.0, 20.0))))
    deg = rng.choice([0, 3, 3, 4, 5, 6, 6, 6, 7, 8])
    pos = rng.randint(1, min(6, n // 8))
    case = dict(kind=kind, n=n, m=m, deg=deg, pos=pos, fp=rng.uniform(0.005, 0.10), fn=rng.uniform(0.02, 0.25),
                q=pos / n)
    sweeps = rng.uniform(2.0, 30.0)
    case["horizon"] = max(1, int(sweeps * n))
    most = min(524288.0, 3e9 / case["horizon"] * min(1.0, 1500.0 / n))
    case["slots"] = _log_int(rng, 64, max(65.0, most))
    if kind == "range":
        case["range"] = _log_int(rng, 32, case["slots"])
    if rng.random() < 0.2 and n >= 100:
        case["n_active"] = n - rng.randint(1, n // 2)
        case["horizon"] = max(1, int(sweeps * case["n_active"]))
    na = case.get("n_active", n)
    option = rng.choice(["", "", "", "uncoupled", "systematic", "uniform", "lag", "start", "custom"])
    if option == "uncoupled":
        case["coupled"] = False
    elif option == "systematic":
        case.update(coupled=False, scan=mcpd.MCPD_SCAN_SYSTEMATIC)
    elif option == "uniform":
        case["scan"] = mcpd.MCPD_SCAN_UNIFORM
    elif option == "lag":
        case["lag"] = rng.randint(2, na)
    elif option == "start":
        case["init"] = True
    elif option == "custom":
        case.update(custom=True, init=True)
    # a drawn instance may mix slowly: as in the paper's runs, a pair stops at 20 sweeps
    if case.get("coupled", True):
        case["cap"] = 20 * na
    return case


def _design(rng, n, m, deg):
    """Each clone's pools, distinct and ascending: `deg` of them, or two to eight (deg 0)."""
    most = min(deg or 8, m)
    picks = np.sort(rng.integers(0, m, (n, most)), axis=1)
    while True:
        bad = np.flatnonzero((np.diff(picks, axis=1) == 0).any(axis=1))
        if not len(bad):
            break
        picks[bad] = np.sort(rng.integers(0, m, (len(bad), most)), axis=1)
    size = np.full(n, most) if deg else rng.integers(min(2, most), most + 1, n)
    if not deg:
        picks = np.take_along_axis(picks, np.argsort(rng.random((n, most)), axis=1), axis=1)
    keep = np.arange(most)[None, :] < size[:, None]
    picks = np.where(keep, picks, m)
    picks.sort(axis=1)
    ptr = np.concatenate([[0], np.cumsum(size)]).astype(np.int32)
    return ptr, picks[picks < m].astype(np.int32)


def _instance(rng, n, m, deg, pos, fp, fn, q):
    ptr, pools = _design(rng, n, m, deg)
    latent = np.zeros(m, dtype=bool)
    for i in rng.choice(n, pos, replace=False):
        latent[pools[ptr[i]:ptr[i + 1]]] = True
    u = rng.random(m)
    y = np.where(latent, u < 1.0 - fn, u < fp).astype(np.uint8)
    return SimpleNamespace(n=n, m=m, clone_ptr=ptr, clone_pools=pools, y=y, fp=fp, fn=fn, q=q)


def _instances(case, seed, noise=None):
    """`count` instances of n_lo to n_hi clones; with `noise`, all of six pools per clone at that
    noise (what the model is trained on), else of four to eight pools at mixed noise.  The sizes are
    the case's; the seed draws the designs and the outcomes."""
    rng = np.random.default_rng([seed, case["count"], case["n_lo"], case["n_hi"]])
    sizes = np.random.default_rng(case["count"]).integers(case["n_lo"], case["n_hi"] + 1, case["count"])
    out = []
    for n in sizes.tolist():
        m = max(8, int(round(n / 13.0)))
        deg = 6 if noise else int(rng.integers(4, 9))
        pos = 3 if noise else int(rng.integers(1, 7))
        fp, fn = noise or (float(rng.uniform(0.005, 0.1)), float(rng.uniform(0.02, 0.25)))
        out.append(_instance(rng, n, m, deg, pos, fp, fn, pos / n))
    return out


def _eta(inst):
    """Naive log score of every clone."""
    lam = math.log(inst.q) - math.log(1.0 - inst.q)
    a_pos = math.log(1.0 - inst.fn) - math.log(inst.fp)
    a_neg = math.log(inst.fn) - math.log(1.0 - inst.fp)
    owner = np.repeat(np.arange(inst.n), np.diff(inst.clone_ptr))
    npos = np.bincount(owner, weights=inst.y[inst.clone_pools], minlength=inst.n)
    return lam + npos * a_pos + (np.diff(inst.clone_ptr) - npos) * a_neg


def _params(case, seed, inst):
    na = case.get("n_active", 0)
    kw = dict(slots=case["slots"], horizon=case["horizon"], seed=seed, n_active=na,
              scan=case.get("scan", mcpd.MCPD_SCAN_SCORE), coupled=case.get("coupled", True),
              meeting_cap=case.get("cap", 0), lag=case.get("lag", 0))
    if "window_sweeps" in case:
        ell = case["window_sweeps"] * na
        kw.update(k=int(np.round(0.1 * ell)) + 1, ell=ell)
    if case.get("init") or case.get("custom"):
        eta = np.sort(_eta(inst))[-na:] if na else _eta(inst)
        nu = 1.0 / (1.0 + np.exp(1.0 - eta))
        if case.get("custom"):
            kw.update(scan=mcpd.MCPD_SCAN_CUSTOM, scan_weights=0.5 * nu / nu.sum() + 0.5 / len(nu))
        if case.get("init"):
            kw["init_marginals"] = np.where(nu < 0.02, 0.0, nu)
    return kw


def _doubles(n):
    return torch.zeros(n, dtype=torch.float64, device=DEVICE)


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(kind=kind)
    if kind in ("grad", "inputs"):
        s.ctx = mcpd.Context(0)
        s.insts = _instances(case, seed, noise=HIGH)
        s.seg = learned.segments(s.insts)
        s.model = learned.MLP(s.ctx, seed=seed % 1000)
        if kind == "grad":
            s.X = learned.features(s.ctx, s.insts)
            s.seg_dev = torch.from_numpy(s.seg).to(DEVICE)
            tw, tp = _targets(s.insts, s.seg, seed)
            s.tw, s.tp = torch.from_numpy(tw).to(DEVICE), torch.from_numpy(tp).to(DEVICE)
        return s
    if kind == "batch":
        stream = torch.cuda.Stream(0)              # a graph is captured on a stream of its own
        s.ctx = mcpd.Context(0, stream=stream)
        s.insts = _instances(case, seed)
        params = [dict(slots=case["slots"], horizon=case["sweeps"] * i.n, seed=seed + k, instance_id=k,
                       meeting_cap=case["cap_sweeps"] * i.n) for k, i in enumerate(s.insts)]
        s.job = mcpd.Batch(s.ctx, s.insts, params, order_mode=1)
        s.est, s.se = _doubles(s.job.total_active), _doubles(s.job.total_active)
        torch.cuda.synchronize()
        s.job.capture_graph(s.est, s.se)
        return s
    rng = np.random.default_rng([seed, case["n"], case["m"]])
    s.ctx = mcpd.Context(0)
    s.inst = _instance(rng, case["n"], case["m"], case["deg"], case["pos"], case["fp"], case["fn"], case["q"])
    s.kw = _params(case, seed, s.inst)
    if kind == "decode":
        return s
    s.range = case.get("range", 0)
    s.job = mcpd.Plan(s.ctx, s.inst, **s.kw)
    s.est, s.se = _doubles(s.job.n_active), _doubles(s.job.n_active)
    return s


# What a run counts: whole numbers, the same on every schedule.
COUNTS = ("progress_units", "site_updates", "reps_started", "reps_retained", "reps_aborted",
          "zero_completion_slots", "step_limit_hits", "max_tau", "sum_tau", "tau_over_audit")


def _counts(stats):
    return {k: int(stats[k]) for k in COUNTS}


def run(s):
    if s.kind == "decode":
        out = s.ctx.decode(s.inst, **s.kw)
        return dict(est=out["est"], se=out["se"], active=out["active"], **_counts(out["stats"]))
    if s.kind == "inputs":
        X = learned.features(s.ctx, s.insts)
        w, nu = learned.learned_inputs(s.model, X, s.seg, nu_floor=0.02)
        return dict(features=X, w=w, nu=nu)
    if s.kind == "grad":
        loss, out, dout = s.model.loss_grad(s.X, s.seg_dev, s.tw, s.tp)
        # the loss is a sum over single-precision logits
        return dict(loss=np.float32(loss), out=out, dout=dout, grad=s.model.grad)
    if s.kind == "batch":
        s.job.launch_graph()
    elif s.kind == "range":
        s.job.run_slots_async(s.range, s.est, s.se)
    else:
        s.job.run_async(s.est, s.se)
    return dict(est=s.est, se=s.se, **_counts(s.job.collect(allow_step_limit=True)))


def work(case):
    """Integer operations that the method's definition asks for (a site draw and a threshold per
    pool of the drawn clone, for each chain), or the model's multiply-adds; inputs and outputs once."""
    kind = case["kind"]
    if kind in ("grad", "inputs"):
        rows = case["count"] * (case["n_lo"] + case["n_hi"]) / 2.0
        macs = 16 * 64 + 64 * 64 + 64 * 2
        if kind == "grad":
            return dict(bytes=rows * (64 + 8 + 8 + 8) + 5378 * 6, flops=rows * 2 * macs * 3)
        return dict(bytes=rows * (6 * 4 + 64 + 16) + 5378 * 2, flops=rows * 2 * macs)
    if kind == "batch":
        n = (case["n_lo"] + case["n_hi"]) / 2.0
        draws = case["count"] * case["slots"] * case["sweeps"] * n
        return dict(bytes=case["count"] * n * (6 * 4 + 16), flops=draws * (78 / 2 + 4 + 24 + 4))
    na = case.get("n_active", 0) or case["n"]
    deg = case["deg"] or 5
    unit = case.get("window_sweeps", 1) * na
    slots = case.get("range", 0) or case["slots"]
    chains = 2 if case.get("coupled", True) else 1
    site = 0 if case.get("scan") == mcpd.MCPD_SCAN_SYSTEMATIC else 4
    return dict(bytes=case["n"] * (deg * 4 + 4) + na * 16,
                flops=slots * max(unit, case["horizon"]) * (78 / 2 + site + chains * (2 * deg + 2)))


def _targets(insts, seg, seed):
    """Training targets as the plain decode gives them: marginals near the naive posterior, and
    weights in proportion to them."""
    rng = np.random.default_rng([seed, len(insts)])
    p = np.concatenate([1.0 / (1.0 + np.exp(2.0 - _eta(i))) for i in insts]) * rng.uniform(0.5, 1.0, int(seg[-1]))
    return learned.weight_target(p, seg, mode="positive").astype(np.float32), p.astype(np.float32)


def _features64(inst):
    n = inst.n
    size = np.diff(inst.clone_ptr)
    owner = np.repeat(np.arange(n), size)
    pools, y = inst.clone_pools, inst.y.astype(np.float64)
    per = lambda v: np.bincount(owner, weights=v, minlength=n)  # noqa: E731  (sum over a clone's pools)
    pos = per(y[pools])
    every = (size > 0) & (pos == size)
    pool_size = np.bincount(pools, minlength=inst.m).astype(np.float64)
    in_pool = np.bincount(pools, weights=every[owner].astype(np.float64), minlength=inst.m)
    least = np.full(n, np.inf)
    np.minimum.at(least, owner[y[pools] > 0], in_pool[pools][y[pools] > 0])
    lam = math.log(inst.q) - math.log(1.0 - inst.q)
    a_pos = math.log(1.0 - inst.fn) - math.log(inst.fp)
    a_neg = math.log(inst.fn) - math.log(1.0 - inst.fp)
    d, p = np.maximum(size, 1), np.maximum(pos, 1)
    mean = len(pools) / inst.m
    f = np.zeros((n, 16))
    f[:, 0], f[:, 1], f[:, 2] = size / 8.0, pos / 8.0, (size - pos) / 8.0
    f[:, 3] = pos / d
    f[:, 4] = (lam + pos * a_pos + (size - pos) * a_neg) / 10.0
    f[:, 5] = per(pool_size[pools]) / d / mean
    f[:, 6] = per(pool_size[pools] * y[pools]) / p / mean
    f[:, 7] = every
    f[:, 8] = np.where(pos > 0, least, 0.0) / 10.0
    f[:, 9] = per(y[pools] / np.maximum(in_pool[pools], 1.0)) / p
    f[:, 10] = np.where(every, per(y[pools] * (in_pool[pools] == 1)), 0.0) / 8.0
    f[:, 11] = per(y[pools] * (in_pool[pools] == 0)) / 8.0
    f[:, 12] = every.sum() / 100.0
    f[:, 13], f[:, 14], f[:, 15] = lam / 10.0, a_pos / 10.0, a_neg / 10.0
    return f


def exact(case, seed):
    """The learned model in 64 bits.  A decode has no such value: its estimate is a whole-number
    sum over the sampler's own random draws, and is compared bit by bit instead."""
    if case["kind"] not in ("grad", "inputs"):
        return None
    s = prepare(case, seed)
    bits = s.model.W.to(torch.int32) & 0xFFFF
    theta = (bits << 16).view(torch.float32).double().requires_grad_(case["kind"] == "grad")
    if case["kind"] == "grad":
        X = s.X.double()
    else:
        F = np.concatenate([_features64(i) for i in s.insts])
        X = torch.from_numpy(F).to(DEVICE).float().double()        # the model reads single precision
    W1, b1, W2, b2, W3, b3 = torch.split(theta, [1024, 64, 4096, 64, 128, 2])
    h = torch.relu(X @ W1.view(64, 16).T + b1)
    h = torch.relu(h @ W2.view(64, 64).T + b2)
    out = h @ W3.view(2, 64).T + b3
    if case["kind"] == "grad":
        out.retain_grad()
    loss, w, nseg = 0.0, [], len(s.seg) - 1
    for a, b in zip(s.seg[:-1].tolist(), s.seg[1:].tolist()):
        o1, o2 = out[a:b, 0], out[a:b, 1]
        if case["kind"] == "inputs":
            w.append(0.5 * torch.softmax(o1, 0) + 0.5 / (b - a))
            continue
        loss = loss - (s.tw[a:b].double() * torch.log_softmax(o1, 0)).sum() / nseg
        loss = loss + torch.nn.functional.binary_cross_entropy_with_logits(o2, s.tp[a:b].double()) / nseg
    if case["kind"] == "inputs":
        nu = torch.sigmoid(out[:, 1]).clamp(1e-6, 1.0 - 1e-6)
        nu = torch.where(nu < 0.02, torch.zeros_like(nu), nu)
        return dict(features=F, w=torch.cat(w), nu=nu)
    loss.backward()
    return dict(loss=float(loss), out=out.detach(), dout=out.grad, grad=theta.grad)
