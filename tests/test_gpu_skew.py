"""The skewed engines (csrc/skew.cuh) at its edges, against the CPU oracle: reads of one
row and around the team's and the strip's start and end (a lane starts one step after its
left neighbour), widths around multiples of a lane and of a strip, gcp Phred 10 throughout
(a constant of the code) and other or mixed values, insertion qualities that jump between rows.

Tolerance: the library's own a-priori FP32 bound for the pair, (6.5 sqrt(16 l + 4 k) 2^-23 +
8 l 2^-46) / ln 10, plus one rounding of log10 L.  No pair may need the FP64 pass."""
import numpy as np
import pytest

import oracle
from paper_2606_25738_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def phmm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_25738_gb300 import phmm as P
    return P


def _pairs(shapes, gcp, ins, seed):
    rng = np.random.default_rng(seed)
    out = []
    for l, k in shapes:
        hap = rng.choice(list(b"ACGT"), size=max(k, l)).astype(np.uint8)
        read = hap[:l].copy()
        m = rng.random(l) < 0.02
        read[m] = rng.choice(list(b"ACGTN"), size=int(m.sum()))
        i = np.arange(l)
        g = {"ten": 10, "other": 13, "mixed": i % 7 + 7}[gcp]
        q = {"flat": 45, "jumps": i * 7 % 30 + 20}[ins]
        out.append((read.tobytes(), hap[:k].tobytes(), rng.integers(8, 41, l), q, 44, g))
    return W.from_strings(out)


def _check(phmm, b, copies=1, **kw):
    pick = np.arange(len(b["pair_read"]))
    with phmm.Context(precision="fp32", **kw) as ctx:
        out, flags, rc, st = ctx.run(W.subset(b, np.tile(pick, copies)) if copies > 1 else b)
    ref = np.tile(oracle.batch(b), copies)
    l, k = (np.tile(x, copies) for x in W.pair_lengths(b))
    tol = (6.5 * np.sqrt(16.0 * l + 4.0 * k) * 2.0 ** -23 + 8.0 * l * 2.0 ** -46) / np.log(10.0) + np.abs(ref) * 2.0 ** -52
    assert rc == 0 and not np.any(flags & 0x79)
    assert np.all(np.abs(out - ref) <= tol), np.max(np.abs(out - ref) / tol)
    return st


@pytest.mark.parametrize("gcp,ins", [("ten", "flat"), ("ten", "jumps"), ("other", "jumps"), ("mixed", "flat")])
@pytest.mark.parametrize("copies", [1, 120])  # a warp for each pair; more pairs than warps: teams
@pytest.mark.parametrize("N,variant", [(32, "pipe2"), (24, "pipe2"), (32, "pipe2lean")])
def test_short_teams(phmm, N, variant, gcp, ins, copies):
    w = 32 * N
    shapes = [(1, 1), (1, w), (2, N), (2, N + 1), (3, 2 * N - 1), (31, w), (32, w - 1), (33, w), (34, w - N), (35, 5),
              (64, N * 16), (65, N * 16 + 1), (150, 431), (151, 250), (300, w), (700, 3 * N), (40, 256), (97, 257), (96, 513)]
    st = _check(phmm, _pairs(shapes, gcp, ins, 5), copies, variant=variant, cols_per_lane=N)
    assert st["short_kernel"] == {("pipe2", 32): 7, ("pipe2", 24): 8, ("pipe2lean", 32): 9}[variant, N]


@pytest.mark.parametrize("gcp,ins", [("ten", "flat"), ("ten", "jumps"), ("other", "jumps"), ("mixed", "flat")])
@pytest.mark.parametrize("kind", ["serial", "wave", "wave16"])
def test_strips(phmm, kind, gcp, ins):
    flag = {"serial": phmm.F_LONG_SERIAL, "wave": phmm.F_LONG_WAVE, "wave16": phmm.F_LONG_WAVE16}[kind]
    shapes = [(1, 1025), (2, 1025), (3, 2048), (16, 2049), (17, 3072), (31, 1536), (32, 1537), (33, 4097), (34, 2080),
              (63, 5000), (64, 1100), (65, 3000), (96, 1056), (97, 1057), (400, 7000), (1500, 1100), (2000, 4100)]
    st = _check(phmm, _pairs(shapes, gcp, ins, 6), flags=flag)
    assert st["long_kernel"] in {"serial": (3,), "wave": (6, 7, 8), "wave16": (8,)}[kind]


# FP64: every path through the matrices adds positive terms, with at most 16 roundings (2^-53 each)
# per row or column in the engine and as many in the oracle, plus one of log10 L
@pytest.mark.parametrize("gcp,ins", [("ten", "flat"), ("other", "jumps"), ("mixed", "flat")])
@pytest.mark.parametrize("variant", [4, 5])
def test_short_teams_fp64(phmm, variant, gcp, ins):
    N = {4: 16, 5: 32}[variant]
    w = 32 * N
    shapes = [(1, 1), (1, w), (2, N), (2, N + 1), (3, 2 * N - 1), (31, w), (32, w - 1), (33, w), (34, w - N), (35, 5),
              (64, N * 16), (65, N * 16 + 1), (150, 431), (700, 3 * N), (1500, 90)]
    b = _pairs(shapes, gcp, ins, 5)
    with phmm.Context(precision="fp64", variant={4: "pipe", 5: "pipe2"}[variant]) as ctx:
        out, flags, rc, st = ctx.run(b)
    ref = oracle.batch(b)
    l, k = W.pair_lengths(b)
    tol = 32.0 * (l + k) * 2.0 ** -53 / np.log(10.0) + np.abs(ref) * 2.0 ** -51
    assert rc == 0 and not np.any(flags & 0x79) and st["short_kernel"] == {4: 2, 5: 3}[variant]
    assert np.all(np.abs(out - ref) <= tol), np.max(np.abs(out - ref) / tol)


@pytest.mark.parametrize("gcp,ins", [("ten", "flat"), ("other", "jumps"), ("mixed", "flat")])
@pytest.mark.parametrize("variant", ["pipe", "pipe2"])
def test_strips_fp64(phmm, variant, gcp, ins):
    shapes = [(1, 1025), (2, 1025), (3, 1280), (16, 1281), (17, 3072), (31, 1536), (32, 1537), (33, 4097), (34, 2080),
              (63, 5000), (64, 1100), (65, 3000), (96, 1056), (97, 1057), (400, 7000), (1500, 1100), (2000, 4100), (60, 900)]
    b = _pairs(shapes, gcp, ins, 6)
    with phmm.Context(precision="fp64", variant=variant) as ctx:
        need = ctx.footprint(b)
        out, flags, rc, st = ctx.run(b)
    ref = oracle.batch(b)
    l, k = W.pair_lengths(b)
    tol = 32.0 * (l + k) * 2.0 ** -53 / np.log(10.0) + np.abs(ref) * 2.0 ** -51
    assert rc == 0 and not np.any(flags & 0x79) and st["n_long"] == len(shapes) - (1 if variant == "pipe2" else 0)
    assert np.all(np.abs(out - ref) <= tol), np.max(np.abs(out - ref) / tol)
    # the footprint's bound is enough, whichever strips fit in it
    with phmm.Context(precision="fp64", variant=variant, mem_budget=need) as ctx:
        small = ctx.run(b)[0]
    assert np.all(np.abs(small - ref) <= tol)


def test_degenerate_strips_fp64(phmm):
    """gcp Phred 0 (T_DD = 1), which the strips cannot hold: a wide pair's flags stay those of
    the unfactored engine."""
    b = _pairs([(50, 2000), (200, 1500)], "other", "flat", 3)
    b["gcp_q"] = np.zeros_like(b["gcp_q"])
    with phmm.Context(precision="fp64", variant="pipe2") as ctx:
        out, flags, rc, st = ctx.run(b)
    with phmm.Context(precision="fp64", cols_per_lane=8) as ctx:
        out8, flags8, _, _ = ctx.run(b)
    assert rc == 0 and np.array_equal(flags, flags8) and np.array_equal(out, out8)


@pytest.mark.parametrize("shape", [(3, 1025), (2, 1000)])
@pytest.mark.parametrize("n", [1, 607, 609, 1217, 1825])
def test_items_around_the_warps(phmm, shape, n):
    """Items one fewer and one more than the warps that are first on their SM, second, all."""
    st = _check(phmm, _pairs([shape] * n, "ten", "flat", 2), flags=phmm.F_LONG_SERIAL, variant="pipe2", cols_per_lane=32)
    assert st["n_long"] == (n if shape[1] > 1024 else 0)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_tags_start_over(phmm, precision):
    """Boundary rows carry one of 63 tags, stepped at every launch.  140 launches on one slot, two
    batches by turns, so that a row's tag comes back under the other batch's layout, whose row it
    must not pass for."""
    bs = [_pairs(shapes, "mixed", "jumps", s) for s, shapes in
          ((7, [(90, 5000), (33, 1100), (150, 2600)]), (8, [(40, 1300), (200, 4200), (17, 1025), (77, 3000)]))]
    kw = dict(flags=phmm.F_LONG_WAVE16) if precision == "fp32" else dict(variant="pipe2")
    with phmm.Context(precision=precision, max_inflight=1, **kw) as ctx:
        first = [ctx.run(b)[0] for b in bs]
        for i in range(138):
            out, flags, rc, st = ctx.run(bs[i % 2])
            assert rc == 0 and np.array_equal(out, first[i % 2]), i
    for b, out in zip(bs, first):
        assert np.max(np.abs(out - oracle.batch(b))) <= {"fp32": 1e-3, "fp64": 1e-9}[precision]
