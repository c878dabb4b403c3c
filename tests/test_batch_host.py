"""A batch's launches as the library's host code makes them, on the stand-in runtime of
tests/fake_cuda (no GPU): every slot lies in exactly one chunk, no chunk exceeds the bank its
scratch is laid out for, none is empty, and the scratch holds every warp's part."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import synth
from paper_2608_30239_gb300 import build, mcpd
from test_gpu_batch_chunks import CASES, small_chunks

HERE = os.path.dirname(os.path.abspath(__file__))
PAIR_STATS = 10


class Host:
    def __init__(self, lib):
        self.lib = lib
        for name, res, args in (("fake_budget", None, [C.c_int64]), ("fake_allocs", None, [C.c_int64]),
                                ("fake_live", C.c_int64, []),
                                ("fake_device", C.c_int, [C.c_int]), ("fake_stage", None, [C.c_void_p]), ("fake_clear_log", None, []),
                                ("fake_log", C.c_int64, [C.c_void_p, C.c_int64])):
            f = getattr(lib, name)
            f.restype, f.argtypes = res, args
        self.ctx = mcpd.Context(0, stream=1)

    def run(self, batch, call="mcpd_batch_run_async", *args):
        """Status, and the launches: dicts of what each was given."""
        out = np.zeros(max(1, batch.total_active))
        self.lib.fake_clear_log()
        p = out.ctypes.data
        rc = getattr(mcpd.lib(), call)(self.ctx.h, batch.h, *args, p, p)
        return rc, self.launches()

    def launches(self):
        n = self.lib.fake_log(None, 0)
        v = np.zeros(max(n, 1), np.int64)
        self.lib.fake_log(v.ctypes.data, n)
        got, at = [], 0
        while at < n:
            d = dict(zip(("lanes", "grid", "warps", "bank", "units", "n_inst", "words", "marks"), v[at:at + 8].tolist()))
            d["inst"] = v[at + 8:at + 8 + 4 * d["n_inst"]].reshape(-1, 4)       # slots, first chunk, chunks, clones
            at += 8 + 4 * d["n_inst"]
            got.append(d)
        return got


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libmcpd_fake.so")
    inc = ["-I" + build.INCLUDE, "-I" + build.SRC, "-I" + os.path.join(build._cuda_home(), "include")]
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-ffp-contract=off", "-Wl,-Bsymbolic"] + inc +
                          [os.path.join(build.SRC, "mcpd_api.cpp"), os.path.join(build.SRC, "mcpd_tables.cpp"),
                           os.path.join(HERE, "fake_cuda", "fake_cuda.cpp"), "-o", out, "-ldl"])
    kept = mcpd._lib, build.LIB
    mcpd._lib, build.LIB = None, out
    h = Host(mcpd.lib())
    yield h
    h.ctx.close()
    mcpd._lib, build.LIB = kept


def warp_words(bank, na, marks=0, coupled=True):
    return (bank + coupled * min(bank, 16)) * (na + marks) + bank + 32 * PAIR_STATS


def check(launches, slots):
    """Chunks as the kernel cuts them (chunk u of an instance starts at slot u * per)."""
    total = 0
    for d in launches:
        na = int(d["inst"][:, 3].max())
        assert d["grid"] * d["warps"] * warp_words(d["bank"], na, d["marks"]) <= d["words"]
        at = 0
        for P, begin, units, _ in d["inst"].tolist():
            assert begin == at
            at += units
            if P == 0:
                assert units == 0
                continue
            per = -(-P // units)
            assert 0 < per <= d["bank"] and (units - 1) * per < P <= units * per
            total += P
        assert at == d["units"]
    assert total == slots


@pytest.mark.parametrize("name", list(CASES))
def test_more_small_chunks_than_resident_warps(host, name):
    """The batches of tests/test_gpu_batch_chunks.py: on 152 SMs every chunk is smaller than 16 slots,
    more chunks than warps are launched, and the later ones belong to smaller instances."""
    insts, ps = small_chunks(name)
    b = mcpd.Batch(host.ctx, insts, ps, order_mode=1, classes=1)
    rc, got = host.run(b)
    assert rc == 0 and len(got) == 1
    check(got, sum(kw["slots"] for kw in ps))
    d = got[0]
    warps = d["grid"] * d["warps"]
    first_of = np.searchsorted(d["inst"][:, 1], np.arange(d["units"]), side="right") - 1
    clones = d["inst"][first_of, 3]
    assert d["bank"] < 16 and d["units"] > warps == 2432
    assert clones[warps:].max() < clones[:warps].max()
    b.close()


@pytest.mark.parametrize("classes", [0, 1, 3])
@pytest.mark.parametrize("slots", [1, 7, 33, 512, 1000])
def test_every_slot_in_one_chunk(host, slots, classes):
    rng = np.random.default_rng(slots)
    insts = [synth.make_instance(int(n), int(n) // 13, 4 + i % 5, 2, 0.05, 0.1, 2 / n, i, 50 + i)
             for i, n in enumerate(rng.integers(200, 4000, 24))]
    ps = [dict(slots=slots + i % 3, horizon=2 * inst.n, seed=i, instance_id=i) for i, inst in enumerate(insts)]
    b = mcpd.Batch(host.ctx, insts, ps, classes=classes)
    want = sum(kw["slots"] for kw in ps)
    rc, got = host.run(b)
    assert rc == 0
    check(got, want)
    mask = np.array([i % 2 for i in range(len(insts))], np.int32)
    rc, got = host.run(b, "mcpd_batch_extend_async", mask.ctypes.data)
    assert rc == 0
    check(got, sum(kw["slots"] for kw, m in zip(ps, mask) if m))
    b.set_shape(warps_per_block=3)
    rc, got = host.run(b)
    assert rc == 0
    check(got, want)
    b.close()


def _growing(host):
    """Two launches whose scratch grows from 16 warps per block (chunks of 37 slots) to 9 (of 32)."""
    insts = [synth.make_instance(900, 60, 4, 2, 0.05, 0.1, 0.003, i, 50 + i) for i in range(16)]
    ps = [dict(slots=5526, horizon=2 * inst.n, seed=i, instance_id=i) for i, inst in enumerate(insts)]
    b = mcpd.Batch(host.ctx, insts, ps, classes=2)
    rc, got = host.run(b)
    assert rc == 0 and [(d["bank"], d["warps"]) for d in got] == [(37, 16), (37, 16)]
    return b, sum(kw["slots"] for kw in ps)


def _set_shape(host, b, lanes, warps):
    return mcpd.lib().mcpd_batch_set_shape(host.ctx.h, b.h, lanes, warps)


@pytest.mark.parametrize("left", [0, 1, 2])
def test_failed_shape_change(host, left):
    """Memory runs out at the first or the second of two launches, and for good (with two
    allocations the change succeeds): the batch refuses to run, and its graph is gone, until a
    shape is set."""
    b, slots = _growing(host)
    assert host.run(b, "mcpd_batch_capture_graph")[0] == 0
    host.lib.fake_allocs(left)
    try:
        want = 0 if left == 2 else mcpd.MCPD_ENOMEM
        assert _set_shape(host, b, 1, 9) == want
        assert mcpd.lib().mcpd_batch_launch_graph(host.ctx.h, b.h) == mcpd.MCPD_EINVAL
        for call, args in (("mcpd_batch_run_async", ()), ("mcpd_batch_extend_async", (None,)), ("mcpd_batch_capture_graph", ())):
            rc, got = host.run(b, call, *args)
            assert rc == want
            if rc == 0:
                check(got, slots)
    finally:
        host.lib.fake_allocs(-1)
    b.set_shape(9)
    rc, got = host.run(b)
    assert rc == 0 and [(d["bank"], d["warps"]) for d in got] == [(32, 9), (32, 9)]
    check(got, slots)
    b.close()


def test_failed_shape_change_keeps_the_shape(host):
    """Memory for the first launch's larger scratch only: the batch goes on in the shape it had, and
    its launches find no error left over."""
    insts = [synth.make_instance(4000, 100, 4, 2, 0.05, 0.1, 0.003, i, 50 + i) for i in range(8)]
    slots = 8 * 2432
    b = mcpd.Batch(host.ctx, insts, [dict(slots=2432, horizon=12000, seed=i, instance_id=i) for i in range(8)], classes=2)
    rc, got = host.run(b)
    assert rc == 0
    words = [d["words"] for d in got]
    more = 9728 * (2 * 4000 + 125 + PAIR_STATS) - words[0]                      # lane groups of 8, 9728 pairs per launch
    assert 0 < more < words[0]
    host.lib.fake_budget(host.lib.fake_live() + 8 * more * 3 // 2)
    try:
        assert _set_shape(host, b, 8, 0) == mcpd.MCPD_ENOMEM
        assert _set_shape(host, b, 5, 9) == mcpd.MCPD_EINVAL                     # refused before any change
        rc, again = host.run(b)
        assert rc == 0 and [(d["lanes"], d["bank"], d["grid"], d["words"]) for d in again] == \
            [(d["lanes"], d["bank"], d["grid"], d["words"]) for d in got]
        check(again, slots)
    finally:
        host.lib.fake_budget(1 << 40)
    b.set_shape(lanes_per_pair=8)
    assert [d["words"] for d in host.run(b)[1]] == [w + more for w in words]
    b.close()


@pytest.mark.parametrize("part", [0.9, 0.4, 0.1])
def test_batch_in_less_memory(host, part):
    """Where a batch's scratch does not fit, its chunks get smaller: at creation, and for a shape set
    later."""
    insts = [synth.make_instance(n, 60, 4, 2, 0.05, 0.1, 0.003, n, 50 + n) for n in (900, 800, 700, 600)]
    ps = [dict(slots=30000, horizon=2 * inst.n, seed=i, instance_id=i) for i, inst in enumerate(insts)]
    base = host.lib.fake_live()
    b = mcpd.Batch(host.ctx, insts, ps, classes=2)
    rc, got = host.run(b)
    bank, need = [d["bank"] for d in got], host.lib.fake_live() - base
    fixed = need - 8 * sum(d["words"] for d in got)
    b.close()
    host.lib.fake_budget(base + fixed + int(part * (need - fixed)))
    try:
        b = mcpd.Batch(host.ctx, insts, ps, classes=2)
        for warps in (0, 7, 0):
            b.set_shape(warps)
            rc, got = host.run(b)
            assert rc == 0
            check(got, 120000)
            if warps == 0:
                assert all(d["bank"] < was for d, was in zip(got, bank))
        b.close()
        host.lib.fake_budget(base + fixed)
        with pytest.raises(mcpd.McpdError, match="ENOMEM"):
            mcpd.Batch(host.ctx, insts, ps, classes=2)
    finally:
        host.lib.fake_budget(1 << 40)
    assert host.lib.fake_live() == base


@pytest.mark.parametrize("part", [1.0, 0.56, 0.3, 0.05])
def test_plan_in_less_memory(host, part):
    """A plan whose scratch (some 100 sums of n_a words per warp) does not fit gets smaller chunks, for
    all that it fits in: 0.56 of it is what one sum pair per lane (64 per warp) would take."""
    inst = synth.make_instance(1298, 97, 6, 3, 0.1, 0.2, 3 / 1298, 1, 2)
    base = host.lib.fake_live()
    kw = dict(slots=524288, horizon=2000, seed=3)
    plan = mcpd.Plan(host.ctx, inst, **kw)
    need = host.lib.fake_live() - base
    plan.close()
    host.lib.fake_budget(base + int(part * need))
    try:
        plan = mcpd.Plan(host.ctx, inst, **kw)
        out = np.zeros(1298)
        for call, args in (("mcpd_run_async", ()), ("mcpd_run_slots_async", (1000, 0)), ("mcpd_run_slots_async", (700000, 1))):
            host.lib.fake_clear_log()
            assert getattr(mcpd.lib(), call)(host.ctx.h, plan.h, *args, out.ctypes.data, out.ctypes.data) == 0
            d, = host.launches()
            assert 0 < d["units"] <= d["bank"]                                   # a plan logs its chunk there
            assert d["grid"] * d["warps"] * warp_words(d["bank"], 1298) <= d["words"]
        plan.close()
        host.lib.fake_budget(base + need // 1000)
        with pytest.raises(mcpd.McpdError, match="ENOMEM"):
            mcpd.Plan(host.ctx, inst, **kw)
    finally:
        host.lib.fake_budget(1 << 40)
    assert host.lib.fake_live() == base


@pytest.mark.parametrize("n,kw,marks", [
    (2048, dict(k=0, ell=30, horizon=2047), 33), (2048, dict(k=0, ell=30, horizon=2048), 0), (2047, dict(k=0, ell=30, horizon=90), 0),
    (2048, dict(k=0, ell=30, horizon=90, lag=1023), 33), (2048, dict(k=0, ell=30, horizon=90, lag=1024), 0),
    (512, dict(coupled=False, burn=5, length=20, horizon=1023), 9), (512, dict(coupled=False, burn=5, length=20, horizon=1024), 0),
    (511, dict(coupled=False, burn=5, length=20, horizon=0), 0), (512, dict(coupled=False, burn=5, length=2000, horizon=0), 0),
    (2048, dict(k=0, ell=30, horizon=90, trace_stride=1, trace_steps=5), 0)])
def test_marks_rule(host, n, kw, marks):
    """Words of marks (W bit words, two to a word, and one 32-bit word more) where slots are short for their clones, and
    scratch for them."""
    inst = synth.make_instance(n, n // 13, 4, 2, 0.05, 0.1, 2 / n, 1, 2)
    out = np.zeros(n)
    plan = mcpd.Plan(host.ctx, inst, slots=500, seed=3, **kw)
    host.lib.fake_clear_log()
    assert mcpd.lib().mcpd_run_async(host.ctx.h, plan.h, out.ctypes.data, out.ctypes.data) == 0
    d, = host.launches()
    assert d["marks"] == marks
    assert d["grid"] * d["warps"] * warp_words(d["bank"], n, marks, kw.get("coupled", True)) <= d["words"]
    plan.close()
    if "trace_steps" not in kw:
        b = mcpd.Batch(host.ctx, [inst, inst], dict(slots=500, seed=3, **kw))
        rc, got = host.run(b)
        assert rc == 0 and [g["marks"] for g in got] == [marks]
        if kw.get("coupled", True):
            check(got, 1000)
        b.close()


@pytest.mark.parametrize("staged", [False, True])
def test_destroying_a_context_keeps_the_current_device(host, staged):
    live = host.lib.fake_live()
    c = mcpd.Context(0, stream=1)
    if staged:
        host.lib.fake_stage(c.h)
    host.lib.fake_device(1)
    try:
        c.close()
        assert host.lib.fake_device(-1) == 1 and host.lib.fake_live() == live
    finally:
        host.lib.fake_device(0)
