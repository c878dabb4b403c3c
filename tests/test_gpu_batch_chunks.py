"""Batches with more chunks than resident warps, each of fewer than 16 slots, longest slots first: a
warp's next chunk belongs to a smaller instance, and some of its lanes find no slot there (needs a
GB300).  Every instance equals the CPU oracle alone.  tests/test_batch_host.py counts the same
chunks without a GPU."""
import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 1
CASES = {"degree6": (256, 64, 6), "degree8": (256, 100, 8), "mixed": (512, 32, 0)}     # instances, slots, degree


def small_chunks(name):
    """200 to 1500 clones, large and small in turn, horizons in proportion to their clones."""
    count, slots, deg = CASES[name]
    insts, ps = [], []
    for i in range(count):
        n = 200 + (i * 701) % 1301
        m = n // 13
        inst = (synth.make_instance(n, m, deg, 2, 0.05, 0.1, 2 / n, 300 + i, 900 + i) if deg else
                synth.make_mixed_instance(n, m, 2, 7, 2, 0.05, 0.1, 2 / n, 300 + i, 900 + i))
        insts.append(inst)
        ps.append(dict(slots=slots, k=2, ell=20, horizon=n // 20, meeting_cap=2 * n, seed=40 + i, instance_id=i))
    return insts, ps


@pytest.mark.parametrize("name", list(CASES))
def test_next_chunk_of_a_smaller_instance(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_30239_gb300 import build, mcpd
    build.build()
    ctx = mcpd.Context(0, stream=torch.cuda.Stream())
    insts, ps = small_chunks(name)
    b = mcpd.Batch(ctx, insts, ps, order_mode=1, classes=1)
    warps = int(b.info[4] * b.info[5])
    bank = int(b.info[6]) // warps
    assert bank < 16 and sum(-(-kw["slots"] // bank) for kw in ps) > warps       # the case is reached
    est = torch.zeros(b.total_active, dtype=torch.float64, device="cuda:0")
    se = torch.zeros_like(est)
    torch.cuda.synchronize()
    b.run_async(est, se)
    b.collect()
    est, se = est.cpu().numpy(), se.cpu().numpy()
    for i, (inst, kw) in enumerate(zip(insts, ps)):
        M = oracle.Model(inst)
        o = M.run_slots(oracle.coupled_run(2, 20, kw["horizon"], kw["seed"], instance=i, meeting_cap=kw["meeting_cap"]),
                        0, kw["slots"], THREADS)
        e, s = M.finalize(o, kw["slots"], 19)
        got = b.buckets(i)
        for key in ("S1", "S2_lo", "S2_hi", "count"):
            assert np.array_equal(got[key], o[key]), (i, key)
        lo, hi = b.offsets[i], b.offsets[i + 1]
        assert np.array_equal(est[lo:hi], e) and np.array_equal(se[lo:hi], s), i
    b.close()
    ctx.close()
