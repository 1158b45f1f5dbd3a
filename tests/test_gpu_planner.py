"""Batches of many pairs are planned on the device (csrc/planner.cu).  Each pair's result
does not depend on the plan, so the same pairs in batches small enough for the host planner
must give the same bits; the oracle checks a sample.  Shapes: every team width, many run
lengths, wide pairs with one item per pair or per strip, one class only, shared reads; and the
index and offset errors that submit must refuse."""
import numpy as np
import pytest

import oracle
from paper_2606_25738_gb300 import workloads as W

pytestmark = pytest.mark.gpu
HOST = 3000  # pairs of a host plan: more short ones than resident warps, so in teams too


@pytest.fixture(scope="module")
def phmm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_25738_gb300 import phmm as P
    return P


def _batch(l, k, seed, reads=None):
    """reads: number of reads (pairs share them, l[:reads] are their lengths)."""
    rng = np.random.default_rng(seed)
    n, nr = len(k), reads or len(k)
    rl, hl = np.asarray(l[:nr], np.uint64), np.asarray(k, np.uint64)
    roff = np.concatenate([[0], np.cumsum(rl)]).astype(np.uint64)
    hoff = np.concatenate([[0], np.cumsum(hl)]).astype(np.uint64)
    nb, nh = int(roff[-1]), int(hoff[-1])
    acgt = np.frombuffer(b"ACGT", np.uint8)
    return dict(read_bases=acgt[rng.integers(0, 4, nb)], read_off=roff, base_q=rng.integers(10, 41, nb).astype(np.uint8),
                ins_q=rng.integers(40, 46, nb).astype(np.uint8), del_q=np.full(nb, 45, np.uint8),
                gcp_q=np.full(nb, 10, np.uint8), hap_bases=acgt[rng.integers(0, 4, nh)], hap_off=hoff,
                pair_read=(np.arange(n) % nr).astype(np.uint32), pair_hap=np.arange(n, dtype=np.uint32))


def _shapes(name):
    rng = np.random.default_rng(17)
    n = 9000
    if name == "widths":
        return np.full(n, 3), rng.integers(1, 1025, n), None
    if name == "runs":
        return np.rint(np.exp(rng.uniform(0, np.log(700), n))).astype(int), rng.integers(1, 200, n), None
    if name == "wide":
        return rng.integers(1, 20, n), np.rint(np.exp(rng.uniform(np.log(30), np.log(5000), n))).astype(int), None
    if name == "one_class":
        return np.full(n, 20), np.full(n, 100), None
    return np.full(n, 30), rng.integers(1, 1025, n), 40  # shared reads


@pytest.mark.parametrize("kind", ["auto", "serial", "wave", "wave16"])
@pytest.mark.parametrize("name", ["widths", "runs", "wide", "one_class", "shared"])
def test_same_bits_as_host_plans(phmm, name, kind):
    if kind != "auto" and name != "wide":
        pytest.skip("no wide pairs")
    l, k, reads = _shapes(name)
    b = _batch(l, k, 3, reads)
    n = len(k)
    flag = {"auto": 0, "serial": phmm.F_LONG_SERIAL, "wave": phmm.F_LONG_WAVE, "wave16": phmm.F_LONG_WAVE16}[kind]
    d = phmm.to_device(b)
    import torch
    for N in (32, 24):
        kw = dict(precision="fp32", variant="pipe2", cols_per_lane=N, flags=flag | phmm.F_NO_TUNE)
        with phmm.Context(**kw) as ctx:
            out, flags, rc, st = ctx.run(b)
            dout = torch.empty(n, dtype=torch.float64, device="cuda")
            ctx.run(d, out=dout)
            parts = [ctx.run(W.subset(b, np.arange(p, min(p + HOST, n)))) for p in range(0, n, HOST)]
        assert rc == 0 and st["n_pairs"] == n and st["cells"] == W.cells(b)
        assert st["n_long"] == int(np.sum(np.asarray(k) > 32 * N))
        assert np.array_equal(out, dout.cpu().numpy())
        if kind != "auto":  # the untuned choice of a wide kind depends on the batch
            assert np.array_equal(out, np.concatenate([p[0] for p in parts]))
            assert np.array_equal(flags, np.concatenate([p[1] for p in parts]))
        else:
            assert np.max(np.abs(out - np.concatenate([p[0] for p in parts]))) <= 1e-5
        pick = np.random.default_rng(1).choice(n, 300, replace=False)
        assert np.max(np.abs(out[pick] - oracle.batch(W.subset(b, pick)))) <= 1e-3


def test_bad_batches_refused(phmm):
    l, k, _ = _shapes("one_class")
    n = len(k)
    with phmm.Context(precision="fp32") as ctx:
        for what in ("index", "offset", "first", "hap"):
            b = _batch(l, k, 4)
            if what == "index":
                b["pair_read"][n - 1] = n
            elif what == "offset":
                b["read_off"][5000] = b["read_off"][4999]
            elif what == "first":
                b["read_off"][0] = 1
            else:
                b["pair_hap"][17] = 0xffffffff
            with pytest.raises(phmm.PhmmError) as e:
                ctx.run(b)
            assert e.value.status == phmm.PHMM_EINVAL
        out, flags, rc, st = ctx.run(_batch(l, k, 4))
        assert rc == 0 and np.all(np.isfinite(out))


@pytest.mark.parametrize("tuned", [False, True])
def test_small_budget_takes_cta_strips(phmm, tuned):
    """A memory budget that holds neither the waves' boundary rows (4096 x 1000 of 16 bytes) nor
    two boundaries of 1000 rows per resident warp: the strips of a CTA need neither, and the tuner
    does not bring back what did not fit."""
    n, l, k = 4096, 1000, 1100
    b = _batch(np.full(n, l), np.full(n, k), 8, 4)
    with phmm.Context(precision="fp32_only", flags=phmm.F_NO_TUNE) as ctx:
        ref = ctx.run(b)[0]
    with phmm.Context(precision="fp32_only", mem_budget=16 << 20, max_inflight=1, flags=0 if tuned else phmm.F_NO_TUNE) as ctx:
        for _ in range(2):  # what was accepted once is accepted again
            out, flags, rc, st = ctx.run(b)
            assert rc == 0 and st["long_kernel"] == 1
            assert np.max(np.abs(out - ref)) <= 1e-3


@pytest.mark.parametrize("precision", ["fp32_only", "fp64"])
def test_tuner_keeps_to_the_budget(phmm, precision):
    """FP32: the 512-column wave strips need 960 MB of boundary rows, the 1024-column ones 384 MB.
    FP64: waves of the pairs up to 1024 columns, which only variant 2 makes, 290 MB.  Neither
    trial may take what the budget does not hold (64 MB: two megabytes a buffer)."""
    import torch
    if precision == "fp64":
        n, l, k, budget = 3010, 3000, np.concatenate([np.full(3000, 800), np.full(10, 2000)]), 150 << 20
    else:
        n, l, k, budget = 600, 20000, np.full(600, 3000), 500 << 20
    b = _batch(np.full(n, l), k, 9, 10)
    with phmm.Context(precision=precision, mem_budget=budget, max_inflight=1) as ctx:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        out, flags, rc, st = ctx.run(b)
        assert rc == 0 and np.all(np.isfinite(out))
        assert free - torch.cuda.mem_get_info()[0] <= budget + (64 << 20)
        if precision != "fp64":
            assert st["long_kernel"] in (6, 7)


@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("l", [195, 200, 205, 210])
def test_packed_and_separate_copies(phmm, l, where):
    """1000 reads whose host arrays come to a little less and a little more than what goes to the
    device in one copy (1 MiB); twice in a row on one slot, so the plan moves or is reused."""
    n = 1000
    b = _batch(np.full(n, l), np.full(n, 40), l)
    pick = np.arange(0, n, 37)
    ref = oracle.batch(W.subset(b, pick))
    with phmm.Context(precision="fp32", max_inflight=1, flags=phmm.F_NO_TUNE) as ctx:
        small = _batch(np.full(n, 20), np.full(n, 40), 1)
        for x in (b, b, small, b):
            out, flags, rc, st = ctx.run(phmm.to_device(x) if where == "device" else x)
            assert rc == 0
    assert np.max(np.abs(out[pick] - ref)) <= 1e-3


@pytest.mark.parametrize("planned", ["host", "device"])
def test_refused_batch_leaves_no_plan(phmm, planned):
    """A batch over the memory budget between two of the same lengths, on one slot: its plan, of
    more pairs, is not taken for theirs."""
    small = _batch(np.full(100, 60), np.full(100, 200), 5)
    n = {"host": 2000, "device": 5000}[planned]
    big = _batch(np.full(n, 3000), np.full(n, 300), 6)
    with phmm.Context(precision="fp32_only", mem_budget=64 << 20, max_inflight=1, flags=phmm.F_NO_TUNE) as ctx:
        first = ctx.run(small)[0]
        for _ in range(2):
            with pytest.raises(phmm.PhmmError) as e:
                ctx.run(big)
            assert e.value.status == phmm.PHMM_ENOMEM
            out, flags, rc, st = ctx.run(small)
            assert rc == 0 and st["n_pairs"] == 100 and np.array_equal(out, first)


@pytest.mark.parametrize("cols", [12, 16])
def test_same_lengths_other_reads(phmm, cols):
    """Packed teams hold two pairs of one read: a batch of the same lengths whose pairs come in
    another order does not take the earlier batch's teams."""
    b = _batch(np.full(320, 60), np.full(320, 150), 7, 40)
    rng = np.random.default_rng(2)
    order = [np.sort(b["pair_read"]), b["pair_read"], rng.permutation(b["pair_read"])]
    with phmm.Context(precision="fp32", cols_per_lane=cols, variant="packed", max_inflight=1, flags=phmm.F_NO_TUNE) as ctx:
        for pr in order:
            x = dict(b, pair_read=pr.astype(np.uint32))
            out, flags, rc, st = ctx.run(x)
            assert rc == 0 and st["packed_kernel"] >= 0
            assert np.max(np.abs(out - oracle.batch(x))) <= 1e-3


@pytest.mark.parametrize("n", [2400, 4096])
def test_asked_waves_stay_waves(phmm, n):
    """F_LONG_WAVE fixes the wave kinds, also where their boundary rows are beyond what the library
    would take by itself; the budget only decides the width of the strips."""
    b = _batch(np.full(n, 300), np.full(n, 4200), 12, 4)
    ref = oracle.batch(W.subset(b, np.arange(0, n, 200)))
    rows = n * 300 * 16  # bytes a boundary: 4 with strips of 1024 columns, 8 with 512
    for budget, kinds in ((0, (8,)), (6 * rows, (6,))):
        with phmm.Context(precision="fp32_only", mem_budget=budget, flags=phmm.F_LONG_WAVE | phmm.F_NO_TUNE) as ctx:
            out, flags, rc, st = ctx.run(b)
        assert rc == 0 and st["long_kernel"] in kinds
        assert np.max(np.abs(out[::200] - ref)) <= 1e-3


def test_footprint_counts_the_planner(phmm):
    """The device planner's scratch (over 5 MB) is part of a batch's footprint, and a budget that
    holds all but it still takes the batch, planned on the host."""
    n = 5000
    b = _batch(np.full(n, 20), np.full(n, 100), 13)
    with phmm.Context(precision="fp32_only") as ctx:
        below, need = (ctx.footprint(W.subset(b, np.arange(m))) for m in (4095, 4096))
        assert need - below > 5 << 20
        need = ctx.footprint(b)
        ref = ctx.run(b)[0]
    for budget in (need, 7 << 20):
        with phmm.Context(precision="fp32_only", mem_budget=budget) as ctx:
            out, flags, rc, st = ctx.run(b)
        assert rc == 0 and np.array_equal(out, ref)


def test_branch_times_of_alternating_fp64_variants(phmm):
    """One slot, batches that the cost model gives to the variants of one kernel and of two
    branches by turns, replayed from graphs: each batch's branch times are its own."""
    one = _batch(np.full(300, 50), np.full(300, 16), 14)
    two = _batch(np.full(300, 200), np.full(300, 1020), 15)
    with phmm.Context(precision="fp64", max_inflight=1, flags=phmm.F_NO_TUNE) as ctx:
        for _ in range(3):
            st = ctx.run(one)[3]
            assert st["short_kernel"] in (0, 1) and st["ms_branch"] == [st["ms_forward"], 0.0, 0.0]
            st = ctx.run(two)[3]
            assert st["short_kernel"] in (2, 3)
            # its short kernel is shorter than the forward pass, its other branch took a time of its own
            assert 0.0 < st["ms_branch"][0] < st["ms_forward"] and st["ms_branch"][1] == 0.0 < st["ms_branch"][2]


def _long_batch(n=20000, l=6000):
    """n pairs of 8 reads and 8 haplotypes of l bases: about 0.2 s of the serial kernel."""
    b = _batch(np.full(8, l), np.full(8, l), 20)
    i = np.arange(n)
    return dict(b, pair_read=(i % 8).astype(np.uint32), pair_hap=(i // 8 % 8).astype(np.uint32))


def test_polling_in_slices_leaves_the_core(phmm):
    """A long batch polled a millisecond at a time: the thread sleeps, but for the first two milliseconds."""
    import time
    with phmm.Context(precision="fp32", flags=phmm.F_NO_TUNE) as ctx:
        ctx.run(_long_batch())
        t = ctx.submit(_long_batch())
        w0, c0 = time.perf_counter(), time.thread_time()
        while (rc := ctx.poll(t, 1)) == phmm.PHMM_PENDING:
            pass
        wall, cpu = time.perf_counter() - w0, time.thread_time() - c0
    assert rc == 0 and wall > 0.1 and cpu < 0.2 * wall, (wall, cpu)


def test_submit_does_not_wait_for_a_batch_in_flight(phmm):
    """A batch of many pairs from host arrays is planned and uploaded while another one fills the
    GPU: submit waits for copies only."""
    import time
    big = _long_batch()
    rng = np.random.default_rng(21)
    small = [_batch(np.full(5000, 100), rng.integers(50, 1500, 5000), s) for s in (22, 23)]
    with phmm.Context(precision="fp32", max_inflight=2, flags=phmm.F_NO_TUNE) as ctx:
        alone = [ctx.run(b)[0] for b in small]
        for _ in range(2):  # the first round allocates
            t0 = time.perf_counter()
            a = ctx.submit(big)
            t1 = time.perf_counter()
            out = np.empty(5000)
            c = ctx.submit(small[0], out)
            t2 = time.perf_counter()
            assert ctx.poll(a) == 0
            t3 = time.perf_counter()
            assert ctx.poll(c) == 0
            assert np.array_equal(out, alone[0])
        assert t3 - t0 > 0.1 and t2 - t1 < 0.25 * (t3 - t0), (t1 - t0, t2 - t1, t3 - t0)
        # plans of two slots, the second made while the first one's batch runs
        outs = [np.empty(5000) for _ in small]
        for _ in range(3):
            tk = [ctx.submit(b, o) for b, o in zip(small, outs)]
            assert [ctx.poll(t) for t in tk] == [0, 0]
            assert all(np.array_equal(o, x) for o, x in zip(outs, alone))
