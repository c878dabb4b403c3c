"""The sampling kernel's builds that mark the clones a slot touches (slots of fewer steps than two sweeps
from 512 clones uncoupled, of fewer than one, from 2048 clones coupled), against
the CPU oracle (needs a GB300): clone counts on both sides of the rule, pairs that meet before and after the
steps that are marked, caps that stop pairs unmet, lags, random starts, refill, dropped slots, several
chunks a warp, and batches.  Integer sums and finalized doubles are equal."""
import os

import numpy as np
import pytest

import oracle
import synth
import test_gpu_uncoupled_sums as sums
from test_gpu_chunks import _buffers, _check, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 1


def _inst(n, m, deg, fp=0.02, fn=0.05, seed=5):
    return (synth.make_instance(n, m, deg, 4, fp, fn, 4 / n, seed, seed + 1) if deg else
            synth.make_mixed_instance(n, m, 2, 7, 4, fp, fn, 4 / n, seed, seed + 1))


COUPLED = {
    "below": (2047, 160, 6, dict(k=2, ell=30, B=90)),
    "line": (2048, 160, 6, dict(k=2, ell=30, B=90)),
    "mixed": (2500, 190, 0, dict(k=0, ell=16, B=200)),
    "window0": (2049, 160, 3, dict(k=0, ell=0, B=40)),
    "degree8": (2100, 230, 8, dict(k=5, ell=100, B=2000)),
    "late": (2048, 60, 5, dict(k=0, ell=40, B=300, cap=4000)),
    "capped": (2048, 60, 5, dict(k=0, ell=20, B=150, cap=25)),
    "lag": (2111, 160, 6, dict(k=3, ell=50, B=900, lag=120)),
    "lag_cap": (2111, 160, 4, dict(k=3, ell=50, B=600, lag=60, cap=70)),
    "start": (2048, 160, 6, dict(k=1, ell=25, B=100, nu=True)),
}


@pytest.mark.parametrize("case", list(COUPLED))
@pytest.mark.parametrize("slots", [1, 17, 3001])
def test_coupled(ctx, case, slots):  # noqa: F811
    n, m, deg, kw = COUPLED[case]
    if kw.get("nu"):
        kw = dict(kw, nu=np.random.default_rng(4).uniform(0.0, 0.02, n))
    _check(ctx, _inst(n, m, deg), slots=slots, runs=2, **kw)


def test_late_pairs_are_on_both_sides():
    """The case above has pairs that meet within half a sweep, and others after (no GPU needed to say so)."""
    n, m, deg, kw = COUPLED["late"]
    r = oracle.Model(_inst(n, m, deg)).run_slots(oracle.coupled_run(0, 40, 300, 5, meeting_cap=4000), 0, 300, THREADS)
    assert r["stats"]["max_tau"] > n // 2 > r["stats"]["sum_tau"] / r["stats"]["reps"]


def test_many_chunks(ctx):  # noqa: F811
    _check(ctx, _inst(2048, 160, 6), k=1, ell=8, B=24, slots=150001, runs=2)


def test_dropped_slots(ctx):  # noqa: F811
    """Slots that run into their step limit are dropped with what they marked; the others are the oracle's."""
    from paper_2608_30239_gb300 import mcpd
    inst, slots, kw = _inst(2048, 60, 5), 2500, dict(k=0, ell=20, horizon=60, seed=8, step_limit=30)
    M = oracle.Model(inst)
    o = M.run_slots(oracle.coupled_run(0, 20, 60, 8, step_limit=30), 0, slots, THREADS, per_slot=True)
    plan = mcpd.Plan(ctx, inst, slots=slots, record_slots=True, **kw)
    est, se = _buffers(plan.n_active)
    for _ in range(2):
        plan.run_async(est, se)
        st = plan.collect(allow_step_limit=True)
        hits = st["step_limit_hits"]
        assert 0 < hits < slots
        g = plan.buckets()
        assert int(g["count"].sum()) == slots - hits
        if int((o["slot_nstar"] == 0).sum()) == hits:
            for key in sums.KEYS:
                assert np.array_equal(g[key], o[key]), key
    plan.close()


@pytest.mark.parametrize("case", [(511, 4, 40, 0), (512, 4, 40, 0), (700, 0, 25, 130), (5000, 8, 7, 0), (1298, 6, 900, 2400)])
@pytest.mark.parametrize("systematic", [False, True])
@pytest.mark.parametrize("slots", [1, 33, 3001])
def test_uncoupled(ctx, case, systematic, slots):  # noqa: F811
    n, deg, T, horizon = case
    sums.test_uncoupled_sums(ctx, n, deg, systematic, slots, T, horizon)


@pytest.mark.parametrize("coupled", [True, False])
def test_batch(ctx, coupled):  # noqa: F811
    """Instances on both sides of the rule in one launch (it goes by the launch's sums)."""
    from paper_2608_30239_gb300 import mcpd
    ns = [90, 3000, 400, 2600, 1300, 700, 5000, 210]
    insts = [_inst(n, max(8, n // 13), 4 + i % 3, 0.05, 0.1, 60 + i) for i, n in enumerate(ns)]
    ps = [dict(slots=700 + 90 * i, horizon=60 + i, seed=50 + i, instance_id=i, coupled=coupled,
               **(dict(k=2, ell=20, meeting_cap=1500) if coupled else dict(burn=5, length=16))) for i in range(len(ns))]
    for classes in (0, 1):
        b = mcpd.Batch(ctx, insts, ps, classes=classes)
        est, se = _buffers(b.total_active)
        for _ in range(2):
            b.run_async(est, se)
            b.collect()
        b.extend_async(est, se, mask=[i % 2 for i in range(len(ns))])
        b.collect()
        for i, kw in enumerate(ps):
            M = oracle.Model(insts[i])
            run = (oracle.coupled_run(2, 20, kw["horizon"], kw["seed"], instance=i, meeting_cap=1500) if coupled else
                   oracle.uncoupled_run(5, 16, kw["horizon"], kw["seed"], instance=i))
            P = kw["slots"] * (1 + i % 2)
            o = M.run_slots(run, 0, P, THREADS)
            e, s = M.finalize(o, P, 19 if coupled else 16)
            g = b.buckets(i)
            for key in sums.KEYS:
                assert np.array_equal(g[key], o[key]), (i, key)
            lo, hi = b.offsets[i], b.offsets[i + 1]
            assert np.array_equal(est[lo:hi].cpu().numpy(), e) and np.array_equal(se[lo:hi].cpu().numpy(), s)
        b.close()


@pytest.mark.parametrize("coupled", [True, False])
def test_noalloc(ctx, coupled):  # noqa: F811
    from paper_2608_30239_gb300 import mcpd
    inst = _inst(2048, 160, 6)
    kw = dict(slots=2000, horizon=100, seed=3, **(dict(k=2, ell=30) if coupled else dict(coupled=False, burn=4, length=20)))
    plan = mcpd.Plan(ctx, inst, **kw)
    est, se = _buffers(plan.n_active)
    plan.run_async(est, se)
    plan.collect()
    e2, s2 = _buffers(plan.n_active)
    for _ in range(2):
        ctx.decode_noalloc(inst, e2, s2, **kw)
        assert np.array_equal(e2.cpu().numpy(), est.cpu().numpy()) and np.array_equal(s2.cpu().numpy(), se.cpu().numpy())
    plan.close()
