"""Uncoupled chains' sums, added over a chunk's slots before they reach their bucket (needs a GB300): clone
counts around a warp's lanes, one slot, chunks that do not divide by the loads in flight, several
chunks a warp, one and several replications a slot, traced slots.  Integer sums, traced sums and finalized doubles
equal the CPU oracle's."""
import os

import numpy as np
import pytest

import oracle
import synth
from test_gpu_chunks import _buffers, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 1
KEYS = ("S1", "S2_lo", "S2_hi", "count")


@pytest.mark.parametrize("n,deg", [(20, 3), (33, 4), (333, 3), (511, 4), (512, 4), (700, 0), (5000, 8)])
@pytest.mark.parametrize("systematic", [False, True])
@pytest.mark.parametrize("slots,T,horizon", [(1, 9, 0), (33, 40, 0), (3001, 25, 130), (40001, 7, 0), (300, 600, 700)])
def test_uncoupled_sums(ctx, n, deg, systematic, slots, T, horizon):  # noqa: F811
    from paper_2608_30239_gb300 import mcpd
    m = max(8, n // 13)
    inst = (synth.make_instance(n, m, deg, 4, 0.05, 0.1, 4 / n, 5, 6) if deg else
            synth.make_mixed_instance(n, m, 2, 7, 4, 0.05, 0.1, 4 / n, 5, 6))
    scan = mcpd.MCPD_SCAN_SYSTEMATIC if systematic else mcpd.MCPD_SCAN_SCORE
    plan = mcpd.Plan(ctx, inst, coupled=False, scan=scan, burn=T // 3, length=T - T // 3 + 1, horizon=horizon, slots=slots,
                     seed=9, trace_stride=max(1, slots // 7))
    est, se = _buffers(plan.n_active)
    M = oracle.Model(inst, scan=oracle.SCAN_SYSTEMATIC if systematic else oracle.SCAN_SCORE)
    o = M.run_slots(oracle.uncoupled_run(T // 3, T - T // 3 + 1, horizon, 9), 0, slots, THREADS, slot_G=n * slots < 4e6)
    e, s = M.finalize(o, slots, T - T // 3 + 1)
    for _ in range(2):
        plan.run_async(est, se)
        plan.collect()
        g = plan.buckets()
        for key in KEYS:
            assert np.array_equal(g[key], o[key]), key
        assert np.array_equal(est.cpu().numpy(), e) and np.array_equal(se.cpu().numpy(), s, equal_nan=True)
        if o["slot_G"] is not None:
            G = plan.fetch(mcpd.MCPD_FETCH_TRACE_G).reshape(-1, n)
            assert np.array_equal(G, o["slot_G"][::max(1, slots // 7)])
    plan.close()
