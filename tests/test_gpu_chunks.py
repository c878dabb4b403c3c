"""The sampling kernel's chunks of slots against the CPU oracle, at the sizes where they can go wrong
(needs a GB300): one slot; fewer and more slots than pairs (16) and lanes (32) of a warp; several
chunks a warp (more than 96 slots each); windows of zero steps, lags beyond the window, doomed
replications whose events began at once; step limits below the window; and a batch whose launches
are cut by pair state.  Integer outputs and finalized doubles are equal."""
import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 1


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_30239_gb300 import build, mcpd
    build.build()
    c = mcpd.Context(0, stream=torch.cuda.Stream())
    yield c
    c.close()


def _buffers(n):
    import torch
    est = torch.zeros(n, dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    return est, torch.zeros_like(est)


def _check(ctx, inst, k, ell, B, slots, seed=5, nu=None, lag=1, cap=0, runs=1):
    from paper_2608_30239_gb300 import mcpd
    plan = mcpd.Plan(ctx, inst, k=k, ell=ell, horizon=B, slots=slots, seed=seed, init_marginals=nu, lag=lag,
                     meeting_cap=cap, record_slots=True)
    est, se = _buffers(plan.n_active)
    M = oracle.Model(inst, init_marginals=nu)
    o = M.run_slots(oracle.coupled_run(k, ell, B, seed, lag=lag, meeting_cap=cap), 0, slots, THREADS, per_slot=True)
    e, s = M.finalize(o, slots, ell - k + 1)
    for _ in range(runs):                       # a second run finds the scratch as the first left it
        plan.run_async(est, se)
        st = plan.collect()
        g = plan.buckets()
        for key in ("S1", "S2_lo", "S2_hi", "count"):
            assert np.array_equal(g[key], o[key]), key
        assert np.array_equal(plan.fetch(mcpd.MCPD_FETCH_SLOT_NSTAR), o["slot_nstar"])
        assert np.array_equal(plan.fetch(mcpd.MCPD_FETCH_SLOT_S), o["slot_S"])
        assert np.array_equal(est.cpu().numpy(), e) and np.array_equal(se.cpu().numpy(), s, equal_nan=True)
        assert st["reps_retained"] == int(o["slot_nstar"].sum())
    plan.close()


@pytest.mark.parametrize("slots", [1, 2, 15, 17, 33, 1825, 29185, 300001])
def test_slot_counts(ctx, slots):
    _check(ctx, synth.tiny_config(1), 3, 20, 65, slots, runs=2)


@pytest.mark.parametrize("case", ["window0", "window1", "odd", "events_at_once", "lag_beyond", "lag_cap", "start"])
def test_windows_lags_and_starts(ctx, case):
    inst = synth.make_instance(170, 16, 5, 4, 0.15, 0.25, 4 / 170, 61, 62)
    nu = np.random.default_rng(4).uniform(0.0, 0.3, inst.n)
    kw = {"window0": dict(k=0, ell=0, B=40, nu=nu), "window1": dict(k=1, ell=1, B=37),
          "odd": dict(k=9, ell=61, B=200), "events_at_once": dict(k=0, ell=12, B=30),
          "lag_beyond": dict(k=3, ell=20, B=260, lag=33), "lag_cap": dict(k=0, ell=15, B=400, lag=7, cap=90),
          "start": dict(k=2, ell=90, B=300, nu=nu)}[case]
    _check(ctx, inst, slots=3001, **kw)


def test_step_limit_below_the_window(ctx):
    """Every slot runs into a step limit below l and is dropped; the next run of the same plan size
    without it is unaffected."""
    from paper_2608_30239_gb300 import mcpd
    inst = synth.tiny_config(1)
    plan = mcpd.Plan(ctx, inst, k=3, ell=20, horizon=60, slots=700, seed=2, step_limit=13)
    est, se = _buffers(plan.n_active)
    for _ in range(2):
        plan.run_async(est, se)
        st = plan.collect(allow_step_limit=True)
        assert st["status"] == mcpd.MCPD_ESTEP_LIMIT and st["step_limit_hits"] == 700 == st["reps_started"]
        assert st["progress_units"] == 700 * 13 and st["reps_retained"] == 0
        assert not plan.buckets()["count"].any() and not plan.buckets()["S1"].any()
    plan.close()
    _check(ctx, inst, 3, 20, 60, 700, seed=2)


@pytest.mark.parametrize("slots", [1, 31, 2433, 300001])
def test_uncoupled_slot_counts(ctx, slots):
    from paper_2608_30239_gb300 import mcpd
    inst = synth.tiny_config(2)
    plan = mcpd.Plan(ctx, inst, coupled=False, scan=mcpd.MCPD_SCAN_SYSTEMATIC, burn=4, length=16, horizon=70, slots=slots,
                     seed=9)
    est, se = _buffers(plan.n_active)
    plan.run_async(est, se)
    plan.collect()
    g = plan.buckets()
    M = oracle.Model(inst, scan=oracle.SCAN_SYSTEMATIC)
    o = M.run_slots(oracle.uncoupled_run(4, 16, 70, 9), 0, slots, THREADS)
    for key in ("S1", "S2_lo", "S2_hi", "count"):
        assert np.array_equal(g[key], o[key]), key
    plan.close()


def test_batch_cut_into_launches(ctx):
    """Twelve instances of 300 to 5000 clones, 4096 slots each, in automatic classes: more columns than
    the GPU holds at once, so classes are cut into launches.  The small instances equal the oracle's."""
    from paper_2608_30239_gb300 import mcpd
    ns = [300, 5000, 320, 4800, 340, 4700, 360, 4600, 380, 4500, 400, 4400]
    insts = [synth.make_instance(n, n // 13, 4 + i % 3, 3, 0.06, 0.15, 3 / n, 700 + i, 800 + i) for i, n in enumerate(ns)]
    ps = [dict(slots=4096, k=2, ell=40, horizon=90 + i, seed=50 + i, instance_id=i) for i in range(len(ns))]
    b = mcpd.Batch(ctx, insts, ps)
    est, se = _buffers(b.total_active)
    for _ in range(2):
        b.run_async(est, se)
        b.collect()
    for i in range(0, len(ns), 2):
        M = oracle.Model(insts[i])
        o = M.run_slots(oracle.coupled_run(2, 40, 90 + i, 50 + i, instance=i), 0, 4096, THREADS)
        e, s = M.finalize(o, 4096, 39)
        g = b.buckets(i)
        for key in ("S1", "S2_lo", "S2_hi", "count"):
            assert np.array_equal(g[key], o[key]), (i, key)
        assert np.array_equal(est[b.offsets[i]:b.offsets[i + 1]].cpu().numpy(), e)
        assert np.array_equal(se[b.offsets[i]:b.offsets[i + 1]].cpu().numpy(), s)
    b.close()
