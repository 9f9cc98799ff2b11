"""The library's size-dependent paths at the sizes where they can go wrong, against the CPU oracle: whole numbers must be
identical, fp64 quantities within 1e-9 relative (tests/parity.py)."""
import ctypes as C
import gc
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

import oracle as orc
import paper_2605_04478_b200 as ccld
from helpers import MiB, frames_from, make_cols
from parity import compare_cumulative, compare_hang, compare_window, make_pair, same

pytestmark = pytest.mark.gpu


def job(sizes, n_seq, rng, t0=1_000_000_000, spacing=20_000_000, dur=None, ent=None, order="rank"):
    """A communicator per entry of `sizes` over ranks of its own, n_seq ops each: (registry, columns, ranks)."""
    reg, parts, r0 = [], [], 0
    for cid, n in enumerate(sizes):
        d = rng.integers(1_000_000, 1_200_000, (n_seq, n)) if dur is None else dur(cid, n)
        e = rng.integers(0, 40_000, (n_seq, n)) if ent is None else ent(cid, n)
        reg.append((cid, list(range(r0, r0 + n)), 0))
        s, r = np.meshgrid(np.arange(n_seq), np.arange(n), indexing="ij")
        te = t0 + s * spacing + e
        parts.append((r0 + r.T.ravel(), np.full(n * n_seq, cid), s.T.ravel(), te.T.ravel(), (te + d).T.ravel()))
        r0 += n
    rank, comm, seq, te, tx = (np.concatenate(x) for x in zip(*parts))
    i = np.arange(len(rank)) if order == "rank" else rng.permutation(len(rank))
    cols = dict(rank=rank[i].astype(np.uint32), comm=comm[i].astype(np.uint32), seq=seq[i].astype(np.uint32),
                op=np.zeros(len(i), np.uint8), bytes=np.full(len(i), 16 * MiB, np.uint64), t_enter=te[i].astype(np.int64),
                t_exit=tx[i].astype(np.int64), send_chg=rng.integers(0, 9, len(i)).astype(np.uint32),
                recv_chg=rng.integers(0, 9, len(i)).astype(np.uint32))
    return reg, cols, r0


def run(reg, cols, n_ranks, params=None, now=10**13, an=None):
    pair = make_pair(reg, params)
    an, o = (an or pair[0]), pair[1]
    an.trace_upload(0, cols)
    assert o.upload(0, cols) == 0
    an.analyze_window(0, 1, now)
    assert o.analyze(0, 1, now) == 0
    compare_window(an, o, 0)
    compare_cumulative(an, o, n_ranks, 0)
    return an, o


# ---------------------------------------------------------------- reductions
@pytest.mark.parametrize("n", [1025, 2048, 2049, 4096, 4097, 8192])
@pytest.mark.parametrize("spread", ["equal", "ties", "wide"])
def test_large_communicators(n, spread):
    """The three instances of the cluster kernel at both ends of their ranges (an eighth of 1,025 or 2,049 members leaves
    CTAs with uneven shares), with all keys equal, more ties than a bin's list holds, and durations over the whole 32 bits (so
    that the median takes every level of the histogram); nine ops: a full tile and one of a single op."""
    rng = np.random.default_rng(n)
    dur = {"equal": lambda c, n: np.full((9, n), 5_000_000), "ties": lambda c, n: 1_000_000 + rng.integers(0, 3, (9, n)),
           "wide": lambda c, n: rng.integers(1, (1 << 31) - 1, (9, n))}[spread]
    ent = {"equal": lambda c, n: np.zeros((9, n), int), "ties": lambda c, n: rng.integers(0, 2, (9, n)) * 4096,
           "wide": lambda c, n: rng.integers(0, 1 << 31, (9, n))}[spread]
    run(*job([n], 9, rng, dur=dur, ent=ent, spacing=5_000_000_000))


def test_three_sizes_side_by_side_on_a_stream():
    """Small, middle and large communicators in one batch, on a stream of the caller's, analysed again and again: the three
    reductions run on streams of their own and share the lists of set-aside groups and the cumulative sums."""
    rng = np.random.default_rng(3)
    reg, cols, n = job([4, 8, 64, 129, 513, 1024, 1500], 19, rng)
    late = rng.random(len(cols["rank"])) < 0.0005
    cols["t_exit"][late] = -1                                   # groups of every size in flight
    st = torch.cuda.Stream()
    an = ccld.Analyzer(stream=st)
    for cid, ranks, seq0 in reg:
        an.comm_register(cid, ranks, 0, seq0)
    an, o = run(reg, cols, n, an=an)
    for _ in range(20):
        an.reset()
        an.analyze_window(0, 1, 10**13)
        compare_cumulative(an, o, n, 0)
    compare_window(an, o, 0)


@pytest.mark.parametrize("sizes", [(1, 3, 7, 8), (9, 32, 33, 64), (65, 127, 128)])
def test_times_across_a_boundary_of_32_bits(sizes):
    """Ops whose enter times, or whose enter and exit, lie on different sides of a multiple of 2^32 ns."""
    rng = np.random.default_rng(sum(sizes))
    run(*job(sizes, 70, rng, t0=(1 << 32) * 5 - 35 * 1_000_000, spacing=1_000_000))


@pytest.mark.parametrize("n", [129, 256, 257, 512, 513, 1024])
def test_middle_communicators_ragged_tiles(n):
    rng = np.random.default_rng(n)
    run(*job([n, n], 13, rng, dur=lambda c, n: 1_000_000 + rng.integers(0, 5 if c else 200_000, (13, n)), order="shuffled"))


@pytest.mark.parametrize("n_comms", [4096, 4097, 8193])
def test_many_communicators(n_comms):
    """Registries at and beyond what the layout keeps in registers and a slice of the emit pass covers."""
    rng = np.random.default_rng(n_comms)
    run(*job([2] * (n_comms - 3) + [40, 200, 8], 3, rng))


@pytest.mark.parametrize("n", [512, 513, 4096])
def test_op_counts_of_wide_communicators(n):
    """Members of communicators of up to 512 are counted by one warp, of more by four; several of both in a CTA's four."""
    rng = np.random.default_rng(n)
    run(*job([n, 5, n, n, 600, 4], 2, rng))


# ---------------------------------------------------------------- verdicts
@pytest.mark.parametrize("n_ranks,outliers", [(900, 1.0), (1024, 0.9), (1100, 0.2), (2100, 1.0), (5000, 0.1), (5000, 0.9)])
def test_verdict_lists(n_ranks, outliers):
    """Suspect lists of one and of several pieces, put together by the last CTA (up to 1,024 entries) and by the merge; the
    columns and the structs of the two entry points say the same, and a capacity cuts the list off."""
    rng = np.random.default_rng(n_ranks)
    # in every group of five, members that are always late or always slow; with a vote share of nothing every outlier counts
    m = n_ranks // 5
    lag = (rng.random((m, 5)) < 0.25 * outliers) * 3_000_000

    def ent(c, n):
        return rng.integers(0, 1000, (12, n)) + lag[c]

    def dur(c, n):
        return 1_000_000 + rng.integers(0, 1000, (12, n)) + np.roll(lag[c], 1)
    reg, cols, n = job([5] * m, 12, rng, ent=ent, dur=dur)
    an, o = run(reg, cols, n, params=dict(vote_rep_milli=200))
    v = an.get_verdict(0)
    k = v["n_suspects_total"]
    assert len(v["suspects"]["rank"]) == k and len(v["comm_rows"]["comm"]) == m and len(v["alerts"]["seq"]) == 0
    s = ccld.Verdict()
    sus, rows = (ccld.Suspect * max(k, 1))(), (ccld.CommVerdict * m)()
    s.suspects, s.suspects_cap, s.comm_rows, s.comm_rows_cap = sus, k, rows, m
    assert an.lib.ccld_get_verdict(an.h, 0, C.byref(s)) == 0 and s.n_suspects_total == k
    for f, _ in ccld.Suspect._fields_:
        same(v["suspects"][f], [getattr(x, f) for x in sus[:k]], f)
    for f, _ in ccld.CommVerdict._fields_:
        same(v["comm_rows"][f], [getattr(x, f) for x in rows], f)
    few = an.get_verdict(0, comm_rows_cap=3, suspects_cap=k // 2)
    assert len(few["comm_rows"]["comm"]) == 3 and few["n_comm_rows_total"] == m and few["n_suspects_total"] == k
    same(few["suspects"]["rank"], v["suspects"]["rank"][:k // 2], "cut suspects")
    if (n_ranks, outliers) == (5000, 0.9):
        assert k > 1024


def test_what_the_binding_hands_out_outlives_the_context():
    """Tables and statistics lie in pinned blocks that go back when the last array is gone, also after the context; a column
    that is not a plain array takes the general way in; windows that are not there are named in the error."""
    rng = np.random.default_rng(8)
    reg, cols, n = job([700, 8, 3], 150, rng)
    an, o = run(reg, cols, n)
    want = o.groups(0)["t_max"].copy()
    kept = [an.get_optable(0) for _ in range(30)] + [an.get_rank_stats(n) for _ in range(30)]
    with pytest.raises(ccld.CcldError):
        an.get_verdict(7)
    assert an.get_verdict(7, check=False)["rc"] != 0
    an.trace_upload(1, {k: (torch.from_numpy(v) if k == "t_enter" else v[::1]) for k, v in cols.items()})
    an.trace_upload(2, {k: np.repeat(v, 2)[::2] for k, v in cols.items()})       # not contiguous
    an.analyze_window(1, 2, 10**13)
    for w in (1, 2):
        same(an.get_optable(w)["t_max"], want, "t_max of window %d" % w)
    an.close()
    for t in kept[:30]:
        same(t["t_max"], want, "kept table")
    assert int(kept[-1]["ops"].sum()) > 0 and kept[-1]["votes"].shape == (n, 4)
    del t, kept


# ---------------------------------------------------------------- uploads
# bytes of an upload are 45 per record (37 without rates): one piece up to 256 KB, one 1 MB piece, then pieces of 1 MB by workers
@pytest.mark.parametrize("n_rec", [1, 5825, 5826, 23301, 23302, 300_000])
@pytest.mark.parametrize("pinned", [False, True])
def test_uploads(n_rec, pinned):
    rng = np.random.default_rng(n_rec)
    n_seq = (n_rec + 7) // 8
    reg, cols, n = job([8], n_seq, rng, spacing=2_000_000, order="shuffled")
    cols = {k: v[:n_rec].copy() for k, v in cols.items()}
    an, o = make_pair(reg)
    signed = lambda v: v if v.itemsize == 1 else v.view("i%d" % v.itemsize)      # torch columns are signed, bit for bit the same
    up = {k: torch.from_numpy(signed(v)).pin_memory() for k, v in cols.items()} if pinned else cols
    for w in range(3):
        an.trace_upload(w, up)
        assert o.upload(w, cols) == 0
    if not pinned:
        for v in cols.values():
            v[:] = 0                                            # pageable memory was copied by the time the call returned
    an.analyze_window(0, 3, 10**13)
    assert o.analyze(0, 3, 10**13) == 0
    for w in range(3):
        compare_window(an, o, w)


# ---------------------------------------------------------------- diagnosis
@pytest.mark.parametrize("n,kinds", [(200, 47), (200, 60), (3000, 200)])
def test_opset_with_many_tuples(n, kinds):
    """More different tuples than the pass over majority candidates takes before it counts them another way."""
    rng = np.random.default_rng(kinds)
    reg, cols, _ = job([n], 2, rng)
    cols["bytes"][:] = (1 + rng.integers(0, kinds, len(cols["bytes"]))) * MiB
    an, o = make_pair(reg)
    an.trace_upload(0, cols); assert o.upload(0, cols) == 0
    an.analyze_window(0, 1, 10**13); assert o.analyze(0, 1, 10**13) == 0
    for s in (0, 1):
        a, b = an.opset_check(0, 0, s), o.opset_check(0, 0, s)
        for k in ("n_members", "n_present", "n_deviating_total", "majority_count", "op", "bytes"):
            assert a[k] == b[k], (s, k, a[k], b[k])
        same(a["ranks"], b["ranks"], "deviating ranks")


@pytest.mark.parametrize("n", [2048, 2049, 5000])
def test_hang_in_a_large_ring(n):
    """Rings at and beyond what the decision keeps in shared memory: members that never entered (H1), some that completed
    (H2), all hung with counters (H3), and ranks that went on to a later op."""
    rng = np.random.default_rng(n)
    reg, cols, _ = job([n], 5, rng)
    seq, rank = cols["seq"].copy(), cols["rank"].copy()
    keep = ~((seq == 4) & (rank % 7 != 0))                      # only some enter op 4
    keep &= ~((seq == 3) & (rank == 11))                        # one never reports op 3
    cols = {k: v[keep] for k, v in cols.items()}
    seq, rank = cols["seq"], cols["rank"]
    cols["t_exit"][(seq == 1)] = -1                             # all hung in op 1
    cols["t_exit"][(seq == 2) & (rank % 3 != 0)] = -1           # some completed op 2
    ch = 2
    frames = frames_from([(r, 0, 1, [(40 + (r * 7) % 5, 40 + (r * 3) % 4)] * ch) for r in range(n) if r != 5], ch)
    an, o = make_pair(reg)
    an.trace_upload(0, cols, frames, ch); assert o.upload(0, cols, frames, ch) == 0
    an.analyze_window(0, 1, 10**13); assert o.analyze(0, 1, 10**13) == 0
    assert {compare_hang(an, o, 0, 0, s)["cls"] for s in range(5)} == {1, 2, 3}
    for d in an.locate_hangs(0):
        b = o.locate_hang(0, d["comm"], d["seq"])
        assert d["cls"] == b["cls"] and d["n_roots_total"] == b["n_roots"]
        same(d["roots"], b["roots"][:64], "sweep roots")


# ---------------------------------------------------------------- rates
@pytest.mark.parametrize("n_ranks,ticks,steps", [(1, 2048 * 257, "even"), (3, 200_000, "uneven"), (40, 2047, "even"), (300, 64, "gaps")])
def test_rates_by_spacing(n_ranks, ticks, steps):
    """A stream long enough for the scanned prefix (over 256 tiles, more than eight per rank), samples that are not evenly
    spaced (the guess of a tick's place misses), ops that span many tiles and ops in flight; columns that start off a 16-byte
    boundary."""
    rng = np.random.default_rng(ticks)
    MS = 1_000_000
    off = np.arange(n_ranks + 1) * ticks
    one = np.arange(ticks) * MS
    if steps == "uneven":
        one = np.cumsum(rng.integers(1, 4 * MS, ticks))
    elif steps == "gaps":
        one = one + (np.arange(ticks) > ticks // 2) * 500 * MS
    tn = np.tile(one, n_ranks)
    sc, rc = np.cumsum(rng.integers(0, 2, len(tn))), np.cumsum(rng.random(len(tn)) < 0.3)
    n_rec = 4001
    rank = np.sort(rng.integers(0, n_ranks, n_rec))
    te = rng.integers(-5 * MS, int(one[-1]) + 5 * MS, n_rec)
    tx = te + np.where(rng.random(n_rec) < 0.1, rng.integers(0, int(one[-1]) + 1, n_rec), rng.integers(0, 20 * MS, n_rec))
    tx[::37] = -1
    es, er = orc.derive_rates(rank, te, tx, off, tn, sc, rc)
    for skip in (0, 1):
        def put(a, dt):
            t = torch.zeros(len(a) + skip, dtype=torch.from_numpy(np.zeros(0, dt)).dtype, device="cuda")
            t[skip:] = torch.from_numpy(np.ascontiguousarray(a).astype(dt))
            return t[skip:]
        an = ccld.Analyzer()
        s, r = an.derive_rates(put(rank, np.int32), put(te, np.int64), put(tx, np.int64), put(off, np.int64), put(tn, np.int64), put(sc, np.int32), put(rc, np.int32))
        torch.cuda.synchronize()
        same(s.cpu().numpy().view(np.uint32), es, "send"); same(r.cpu().numpy().view(np.uint32), er, "recv")


# bytes of the columns: within what one kernel reads, one piece, several pieces
@pytest.mark.parametrize("n_rec", [5000, 20_000, 60_000])
@pytest.mark.parametrize("pageable", [(), ("rank",), ("comm", "seq", "op", "send_chg")])
def test_upload_of_columns_the_stream_still_writes(n_rec, pageable):
    """Pinned columns that a copy of the stream fills when the upload is called: their contents are those of their turn in the
    stream. Some columns may be pageable; those are read by the call itself."""
    rng = np.random.default_rng(n_rec)
    reg, cols, _ = job([8], n_rec // 8, rng, spacing=2_000_000, order="shuffled")
    an, o = make_pair(reg)
    assert o.upload(0, cols) == 0
    dev, up = {}, {}
    for i, (k, v) in enumerate(cols.items()):
        t = torch.from_numpy(v if v.itemsize == 1 else v.view("i%d" % v.itemsize))
        dev[k] = t.cuda()
        # an odd column lies off a 16-byte boundary
        up[k] = v.copy() if k in pageable else torch.zeros(len(v) + 3, dtype=t.dtype).pin_memory()[3 * (i % 2):][:len(v)]
    torch.cuda.synchronize()
    torch.cuda._sleep(20_000_000)                               # some ten milliseconds of the stream
    for k in up:
        if k not in pageable:
            up[k].copy_(dev[k], non_blocking=True)
    an.trace_upload(0, up)
    for k in pageable:
        up[k][:] = 0
    an.analyze_window(0, 1, 10**13)
    assert o.analyze(0, 1, 10**13) == 0
    compare_window(an, o, 0)


@pytest.mark.parametrize("to_host", [True, False])
def test_a_window_refused_for_its_size_after_one_of_its_shape(to_host):
    """An op counter far beyond the others makes the window need too many slots. Where an earlier window of as many records made
    the library size the results without waiting, the refused window lists nothing either, and the next one is analysed."""
    rng = np.random.default_rng(5)
    reg, cols, _ = job([8, 4], 50, rng)
    far = {k: v.copy() for k, v in cols.items()}
    far["seq"][7] = 3_000_000_000
    got = []
    for speculate in (True, False):
        an = make_pair(reg)[0]
        an.set_speculation(speculate)
        for w, c in enumerate((cols, far, cols)):
            an.trace_upload(w, c)
            an.analyze_window(w, 1, 10**13)
        t = an.get_optable(1, to_host=to_host)
        got.append((t["n_groups"], t["n_slots"], an.get_verdict(1, check=False), an.get_verdict(2)))
    for G, S, v, after in got:
        assert G == 0 and S == 0 and v["rc"] == -8 and v["n_groups"] == 0 and v["n_comm_rows_total"] == 0
        assert all(len(x) == 0 for x in v["comm_rows"].values())
        assert after["n_groups"] == 100 and after["n_complete"] == 100
    for k in ("slow_count", "rounds_total", "t_max", "n_rounds"):
        same(got[0][3]["comm_rows"][k], got[1][3]["comm_rows"][k], k)


def test_large_pageable_upload_on_the_per_thread_stream():
    """The handle cudaStreamPerThread names another stream in every thread: the library's helpers must not copy on theirs."""
    from types import SimpleNamespace
    rng = np.random.default_rng(6)
    reg, cols, n = job([8], 40_000, rng, spacing=2_000_000, order="shuffled")
    an, o = ccld.Analyzer(stream=SimpleNamespace(cuda_stream=2)), orc.Oracle()
    for cid, ranks, seq0 in reg:
        an.comm_register(cid, ranks, 0, seq0)
        assert o.comm_register(cid, ranks, seq0) == 0
    for w in range(3):
        assert o.upload(w, cols) == 0
        up = {k: v.copy() for k, v in cols.items()}
        an.trace_upload(w, up)
        for v in up.values():
            v[:] = 0
        an.analyze_window(w, 1, 10**13)
        assert o.analyze(w, 1, 10**13) == 0
        compare_window(an, o, w)
        if w:
            an.window_release(w)
    compare_cumulative(an, o, n, 0)


def test_device_memory_goes_back_with_its_context():
    """While another context lives, a context that is closed leaves it blocks of no more than 256 MB in all; the last one to go
    leaves nothing."""
    rng = np.random.default_rng(9)
    reg, cols, _ = job([8], 400_000, rng, spacing=2_000_000)

    def passes():
        an = make_pair(reg)[0]
        for w in range(3):
            an.trace_upload(w, cols)
        an.analyze_window(0, 3, 10**13)
        assert an.get_verdict(2)["n_complete"] == 400_000
        return an

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]
    gc.collect()                                                # contexts of earlier tests
    passes().close()                                            # what the process itself keeps is there by now
    first = free()
    other = ccld.Analyzer()
    an = passes()
    held = first - free()
    assert held > 500 << 20
    an.close()
    assert first - free() <= 258 << 20
    other.close()
    assert first - free() <= 2 << 20


def test_results_may_be_dropped_while_a_graph_is_captured():
    """The last array on a pinned block gives it back, and with no context left it is freed: not a step of a capture."""
    gc.collect()                                                # contexts of earlier tests
    rng = np.random.default_rng(10)
    reg, cols, n = job([4], 50, rng)
    an, _ = run(reg, cols, n)
    kept = [an.get_optable(0), an.get_rank_stats(n)]
    an.close()
    x = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        x += 1
        kept.clear()
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2] * 8


@pytest.mark.parametrize("n", [3, 6, 7, 11, 172, 500, 1024])
def test_bus_bandwidth_of_an_op_is_rounded_once_or_twice(n):
    """bytes * num and span * den are whole numbers that fp64 holds: above 128 members their quotient is rounded once (2^-53), up
    to 128 it is a product with a reciprocal, both rounded (2^-52, and 2^-56 for the reciprocal's last step)."""
    rng = np.random.default_rng(n)
    d = np.exp(rng.normal(np.log(2e6), 1.0, (200, n))).astype(np.int64) + 1
    reg, cols, _ = job([n], 200, rng, dur=lambda c, n: d, spacing=1_000_000_000)
    by = np.exp(rng.normal(np.log(32 * MiB), 1.0, 200)).astype(np.uint64)
    cols["bytes"] = by[cols["seq"]]
    an = make_pair(reg)[0]
    an.trace_upload(0, cols)
    an.analyze_window(0, 1, 10**15)
    t = an.get_optable(0)
    want = by.astype(np.longdouble) * (2 * (n - 1)) / (t["span"].astype(np.longdouble) * n)
    off = float(np.abs((t["busbw"].astype(np.longdouble) - want) / want).max())
    assert off <= (2.0 ** -53 if n > 128 else 2.0 ** -52 + 2.0 ** -56) * (1 + 1e-3), off


_LITTLE_MEMORY = """
import resource, sys
import numpy as np
import paper_2605_04478_b200 as ccld
an = ccld.Analyzer()
an.comm_register(0, range(4))
n = 60_000_000
none = np.zeros(n, np.uint64)
pages = int(open("/proc/self/statm").read().split()[0])
resource.setrlimit(resource.RLIMIT_AS, (pages * 4096 + (256 << 20),) * 2)
print("rc", an.lib.ccld_copy_many_to_host(an.h, n, none.ctypes.data, none.ctypes.data, none.ctypes.data))
"""


def test_copies_of_many_arrays():
    """More arrays than one kernel takes; and so many (empty) ones that a list of them would not fit into memory."""
    an = ccld.Analyzer()
    for k in (1, 24, 25, 100):
        src = [torch.randint(0, 255, (7 * i + 1,), dtype=torch.uint8, device="cuda") for i in range(k)]
        out = an._to_host([(t.data_ptr(), t.numel(), np.uint8) for t in src])
        for t, a in zip(src, out):
            same(a, t.cpu().numpy(), "array")
    r = subprocess.run([sys.executable, "-c", _LITTLE_MEMORY], capture_output=True, text=True, cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0 and r.stdout.strip() == "rc 0", (r.returncode, r.stdout, r.stderr[-500:])


# ---------------------------------------------------------------- units, positions, records in their slots
def cut(cols, keep):
    return {k: v[keep].copy() for k, v in cols.items()}


def again(an, o, n_ranks, times=2):
    """The same window analysed again: sized from what the pass before found."""
    for _ in range(times):
        an.reset()
        an.analyze_window(0, 1, 10**13)
        compare_window(an, o, 0)
        compare_cumulative(an, o, n_ranks, 0)


@pytest.mark.parametrize("most", [1, 31, 33, 96, 700, 2500])
def test_units_over_the_chunks(most):
    """Communicators with fewer, as many and more op counters than a unit and than a chunk, up to more units than there are chunks."""
    rng = np.random.default_rng(most)
    sizes = [2, 4, 5, 8, 9, 32, 33, 65, 128]
    reg, cols, n = job(sizes, most, rng)
    limit = np.array([max(1, most // (1 + c % 4) - c % 3) for c in range(len(sizes))])
    cols = cut(cols, cols["seq"] < limit[cols["comm"]])
    an, o = run(reg, cols, n)
    again(an, o, n, 1)


@pytest.mark.parametrize("n_seq", [1, 32, 45])
@pytest.mark.parametrize("min_group", [1, 4])
def test_four_positions(n_seq, min_group):
    """Groups of one to five, complete and not, all of them tested or only those of four and more; ties."""
    rng = np.random.default_rng(10 * n_seq + min_group)
    reg, cols, n = job([1, 2, 3, 4, 5] * 3, n_seq, rng, dur=lambda c, n: 1_000_000 + rng.integers(0, 4, (n_seq, n)), ent=lambda c, n: rng.integers(0, 3, (n_seq, n)))
    cols["op"] = (cols["seq"] % 3).astype(np.uint8)
    cols["bytes"][cols["seq"] % 5 == 1] = 2                     # barriers
    cols["t_exit"][rng.random(len(cols["seq"])) < 0.02] = -1
    cols = cut(cols, rng.random(len(cols["seq"])) >= 0.02)
    an, o = run(reg, cols, n, dict(min_group=min_group))
    again(an, o, n, 1)


@pytest.mark.parametrize("sizes", [[1] * 40, [3] * 1100, [2] * 33 + [130] * 3 + [1100]])
def test_owner_of_a_group_set_aside(sizes):
    """Every op of a few communicators lacks a member: among fewer than 32 x 32 communicators and more, at both ends."""
    rng = np.random.default_rng(len(sizes))
    reg, cols, n = job(sizes, 3, rng)
    lame = np.isin(cols["comm"], [0, 1, 31, 32, 33, len(sizes) // 2, len(sizes) - 1])
    cols["t_exit"][lame & (rng.random(len(lame)) < 0.4)] = -1
    cols["t_exit"][lame & (rng.random(len(lame)) < 0.2)] = 5    # exit before enter
    cols = cut(cols, ~(lame & (rng.random(len(lame)) < 0.2)))
    an, o = run(reg, cols, n)
    again(an, o, n, 1)


MANY = list(range(1, 9)) * 12 + [9, 33, 64, 128]


@pytest.mark.parametrize("rates", [True, False])
@pytest.mark.parametrize("n_seq", [3, 37, 64])
def test_records_in_no_order(n_seq, rates):
    """From the second pass on such a window's records lie in their slots: complete groups, missing members, ops in flight, sizes that
    differ, records of strangers, then as many records in their ranks' order, and mixed again."""
    rng = np.random.default_rng(n_seq)
    reg, cols, n = job(MANY, n_seq, rng, order="shuffled")
    cols["bytes"][rng.random(len(cols["seq"])) < 0.003] += 4
    cols["op"][rng.random(len(cols["seq"])) < 0.003] = 3
    cols["t_exit"][rng.random(len(cols["seq"])) < 0.003] = -1
    cols = cut(cols, rng.random(len(cols["seq"])) >= 0.003)
    if not rates:
        del cols["send_chg"], cols["recv_chg"]
    an, o = run(reg, cols, n)
    again(an, o, n)
    order = np.lexsort((cols["seq"], cols["comm"], cols["rank"]))
    sorted_ = {k: v[order] for k, v in cols.items()}
    for c in (sorted_, sorted_, cols, cols):
        an.window_release(0)
        an.reset()
        an.trace_upload(0, c)
        an.analyze_window(0, 1, 10**13)
        p = make_pair(reg)[1]
        assert p.upload(0, c) == 0 and p.analyze(0, 1, 10**13) == 0
        compare_window(an, p, 0)
        compare_cumulative(an, p, n, 0)
        an.get_verdict(0)


def test_records_in_no_order_with_strangers():
    """Unknown communicators, ranks that are no members or out of range: rejected and counted as where indices alone are placed."""
    rng = np.random.default_rng(4)
    reg, cols, n = job(MANY, 20, rng, order="shuffled")
    i = rng.choice(len(cols["seq"]), 60, replace=False)
    cols["comm"][i[:20]] = 5000
    cols["comm"][i[20:40]] = 0xFFFFFFFF
    cols["rank"][i[40:50]] = n + 7
    cols["rank"][i[50:]] = 0
    an, o = make_pair(reg)
    an.trace_upload(0, cols)
    o.upload(0, cols)
    an.analyze_window(0, 1, 10**13)
    o.analyze(0, 1, 10**13)
    first = an.get_verdict(0, check=False)
    assert first["n_rejected"] >= 50 and first["n_rejected"] == o.sizes(0)["n_rejected"]
    for _ in range(2):
        an.reset()
        an.analyze_window(0, 1, 10**13)
        compare_window(an, o, 0, expect_rc=first["rc"])


@pytest.mark.parametrize("order", ["rank", "shuffled"])
def test_rows_and_indices_name_the_same_copy_of_a_record(order):
    """Every record twice, the copies differing: whichever wins its slot, the op's row, its flags and the slot's index belong to it."""
    rng = np.random.default_rng(len(order))
    reg, cols, n = job([3, 8, 8, 8, 40] * 60, 100, rng)
    twice = {k: np.concatenate([v, v]) for k, v in cols.items()}
    half = len(cols["seq"])
    twice["t_enter"][half:] += 7_000_000
    twice["t_exit"][half:] += 7_000_000 + rng.integers(1, 9, half) * 1000
    twice["bytes"][half:] += 4
    twice["send_chg"][half:] += 100
    i = rng.permutation(2 * half) if order == "shuffled" else np.lexsort((twice["t_enter"], twice["seq"], twice["comm"], twice["rank"]))
    cols = {k: v[i] for k, v in twice.items()}
    an = make_pair(reg)[0]
    an.trace_upload(0, cols)
    for _ in range(12):
        an.reset()
        an.analyze_window(0, 1, 10**13)
        v = an.get_verdict(0, check=False)
        assert v["rc"] == -10 and v["n_rejected"] == half and v["n_complete"] == v["n_groups"]
        t, r = an.get_optable(0), an.get_ranges(0)
        n_seq = r["n_seq"].astype(np.int64)
        for g0, s0, k, ns in zip(np.cumsum(n_seq) - n_seq, r["slot0"].astype(np.int64), r["n"].astype(np.int64), n_seq):
            at = t["perm"][s0:s0 + k * ns].reshape(k, ns)
            te, du = cols["t_enter"][at], cols["t_exit"][at] - cols["t_enter"][at]
            same(t["e_min"][g0:g0 + ns], te.min(0), "e_min")
            same(t["t_max"][g0:g0 + ns], du.max(0), "t_max")
            same(t["t_min"][g0:g0 + ns], du.min(0), "t_min")
            same(t["max_chg"][g0:g0 + ns], np.maximum(cols["send_chg"][at], cols["recv_chg"][at]).max(0), "max_chg")
            by = cols["bytes"][at]
            same(t["gflags"][g0:g0 + ns] & 8 != 0, (by != by[0]).any(0), "sizes differ")


def in_turn(n_ranks, fams, n_seq, rng, order):
    """Ranks that are in several communicators (groups of `fams[i]` neighbours each) and take turns over them."""
    reg, parts = [], []
    for n in fams:
        for r0 in range(0, n_ranks, n):
            reg.append((len(reg), list(range(r0, r0 + n)), 0))
            r, s = np.meshgrid(np.arange(r0, r0 + n), np.arange(n_seq), indexing="ij")
            parts.append((r.ravel(), np.full(r.size, reg[-1][0]), s.ravel()))
    rank, comm, seq = (np.concatenate(x) for x in zip(*parts))
    i = np.lexsort((comm, seq, rank)) if order == "rank" else rng.permutation(len(rank))
    rank, comm, seq = rank[i], comm[i], seq[i]
    te = 1_000_000_000 + seq * 20_000_000 + rng.integers(0, 40_000, len(i))
    return reg, dict(rank=rank.astype(np.uint32), comm=comm.astype(np.uint32), seq=seq.astype(np.uint32), op=np.zeros(len(i), np.uint8),
                     bytes=np.full(len(i), 16 * MiB, np.uint64), t_enter=te, t_exit=te + rng.integers(1_000_000, 1_200_000, len(i)),
                     send_chg=rng.integers(0, 9, len(i)).astype(np.uint32), recv_chg=rng.integers(0, 9, len(i)).astype(np.uint32)), n_ranks


ORDERS = {  # what, whether its records go to their slots
    "small groups in arrival order": (lambda rng: job([8] * 60, 40, rng, order="shuffled"), True),
    "small groups, rank by rank": (lambda rng: job([8] * 60, 40, rng), False),
    "larger rings, three in ten records of small groups": (lambda rng: job([256] * 16 + [8] * 220, 30, rng, order="shuffled"), False),
    "larger rings, six in ten records of small groups": (lambda rng: job([256] * 16 + [8] * 800, 30, rng, order="shuffled"), True),
    "twelve communicators in turn, rank by rank": (lambda rng: in_turn(64, [8] * 12, 40, rng, "rank"), False),
    "twelve communicators in turn, in arrival order": (lambda rng: in_turn(64, [8] * 12, 40, rng, "shuffled"), True),
    "few ops of many ranks, rank by rank": (lambda rng: in_turn(512, [8, 16, 32, 64] * 3, 5, rng, "rank"), False),
}


@pytest.mark.parametrize("what", list(ORDERS))
def test_which_records_go_to_their_slots(what):
    """Only those in another order than their ranks', and only where the kernel that reads them there has half of the slots and more."""
    make, packed = ORDERS[what]
    reg, cols, n = make(np.random.default_rng(len(what)))
    an, o = run(reg, cols, n)
    again(an, o, n)
    assert an.get_route_counts() == {"unwaited": 2, "redone": 0, "packed": 2 if packed else 0, "filled_under_range": 0}


def test_the_order_of_the_records_is_learned_from_batches_nobody_asks_about():
    """Analysed and reset, again and again, with a window of the shape in another order uploaded in between: the batch after the first
    in the new order goes the other way."""
    rng = np.random.default_rng(16)
    reg, cols, n = job([8] * 60, 40, rng)
    i = rng.permutation(len(cols["seq"]))
    an, o = run(reg, cols, n)
    an.trace_upload(1, {k: v[i] for k, v in cols.items()})
    for w, packed in ((0, 0), (1, 0), (1, 1), (1, 2), (0, 3), (0, 3)):
        an.reset()
        an.analyze_window(w, 1, 10**13)
        assert an.get_route_counts()["packed"] == packed
    again(an, o, n, 1)


def test_records_in_their_slots_keep_their_space_until_the_kernels_are_through():
    """One thread's batch waits on its cudaStreamPerThread while another thread, whose stream is not behind it, uploads windows of about
    the size of that space: the batch's records and the uploads do not meet."""
    from types import SimpleNamespace
    rng = np.random.default_rng(14)
    reg, cols, n = job([8] * 60, 500, rng, order="shuffled")    # 240,000 records: 7.7 MB in their slots
    some = cut(cols, np.sort(rng.permutation(len(cols["seq"]))[:160_000])) # 7.2 MB of columns
    an, o = ccld.Analyzer(stream=SimpleNamespace(cuda_stream=2)), orc.Oracle()
    for cid, ranks, seq0 in reg:
        an.comm_register(cid, ranks, 0, seq0)
        assert o.comm_register(cid, ranks, seq0) == 0
    for w, c in enumerate((cols, some, some, some)):
        assert o.upload(w, c) == 0
    an.trace_upload(0, cols)
    for _ in range(2):
        an.reset()
        an.analyze_window(0, 1, 10**13)
        an.get_verdict(0)
    own = torch.cuda.ExternalStream(2)
    an.reset()
    with torch.cuda.stream(own):
        torch.cuda._sleep(20_000_000)                           # some 10 ms
    an.analyze_window(0, 1, 10**13)

    def upload():
        for w in (1, 2, 3):
            an.trace_upload(w, some)
        torch.cuda.ExternalStream(2).synchronize()
    t = threading.Thread(target=upload)
    t.start()
    t.join()
    assert an.get_route_counts()["packed"] == 2
    assert o.analyze(0, 1, 10**13) == 0
    compare_window(an, o, 0)
    an.analyze_window(1, 3, 10**13)
    assert o.analyze(1, 3, 10**13) == 0
    for w in (1, 2, 3):
        compare_window(an, o, w)
    compare_cumulative(an, o, n, 3)


def test_records_in_their_slots_take_no_more_than_half_of_the_free_memory():
    """A shape whose records do not get their space is gathered, then and later; another shape, with memory there, is not."""
    sizes = [8] * 1600
    cols = device_job(sizes, 800, 15, order="shuffled")         # 10.2 M records, 328 MB in their slots
    an = device_analyzer(sizes)
    an.trace_upload(0, cols)
    an.analyze_window(0, 1, 10**13)
    want = an.get_optable(0)

    def passes(times):
        for _ in range(times):
            an.reset()
            an.analyze_window(0, 1, 10**13)
            got = an.get_optable(0)
            for k in want:
                same(got[k], want[k], k)
        return an.get_route_counts()["packed"]
    gc.collect()
    torch.cuda.empty_cache()
    room = torch.empty(torch.cuda.mem_get_info()[0] - (600 << 20), dtype=torch.uint8, device="cuda")
    assert passes(2) == 0
    del room
    torch.cuda.empty_cache()
    assert passes(2) == 0
    an.window_release(0)
    an.trace_upload(1, {k: v[:-1] for k, v in cols.items()})
    for _ in range(3):
        an.reset()
        an.analyze_window(1, 1, 10**13)
        assert an.get_verdict(1)["n_incomplete"] == 1
    assert an.get_route_counts()["packed"] == 2


# a thread of the uploading kernel has four words of 16 bytes on their way: columns of 4 and 8 bytes around multiples of 1,024 x 4 words
@pytest.mark.parametrize("n_rec", [4095, 4097, 8191, 8192, 8193, 12_289, 16_383, 16_384, 16_387])
def test_pinned_columns_around_the_words_a_kernel_has_in_flight(n_rec):
    test_uploads(n_rec, True)


def test_several_windows_with_records_in_their_slots():
    """A batch of three windows of different record counts, members missing and in flight, with communicators beside them that read
    through the table."""
    rng = np.random.default_rng(17)
    sizes = [3] * 40 + [8] * 100 + [64] * 10 + [200, 1100]      # 1,560 of 2,860 slots per op counter are read where the records lie
    o, wins = None, []
    for w in range(3):
        reg, cols, n = job(sizes, 20 + 13 * w, rng, order="shuffled")
        cols["t_exit"][rng.random(len(cols["seq"])) < 0.002] = -1
        wins.append(cut(cols, rng.random(len(cols["seq"])) >= 0.002))
    an, o = make_pair(reg)
    for w, c in enumerate(wins):
        an.trace_upload(w, c)
        assert o.upload(w, c) == 0
    assert o.analyze(0, 3, 10**13) == 0
    for _ in range(3):
        an.reset()
        an.analyze_window(0, 3, 10**13)
        for w in range(3):
            compare_window(an, o, w)
        compare_cumulative(an, o, n, 2)
    assert an.get_route_counts() == {"unwaited": 2, "redone": 0, "packed": 2, "filled_under_range": 0}


def test_a_captured_batch_gathers():
    """In a graph the space of records in their slots would be shared by whatever is launched beside it: a captured call does without."""
    rng = np.random.default_rng(18)
    reg, cols, n = job([8] * 60, 40, rng, order="shuffled")
    st = torch.cuda.Stream()
    an = ccld.Analyzer(stream=st)
    for cid, ranks, seq0 in reg:
        an.comm_register(cid, ranks, 0, seq0)
    an, o = run(reg, cols, n, an=an)
    again(an, o, n, 1)
    assert an.get_route_counts()["packed"] == 1
    an.reset()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        an.analyze_window(0, 1, 10**13)
    with torch.cuda.stream(st):
        g.replay()
    torch.cuda.synchronize()
    assert an.get_route_counts()["packed"] == 1
    compare_window(an, o, 0)
    compare_cumulative(an, o, n, 0)
    again(an, o, n, 1)
    assert an.get_route_counts()["packed"] == 2


def device_job(sizes, n_seq, seed, order="rank", lost=0):
    """Columns on the GPU: a communicator per entry of `sizes` over ranks of its own, n_seq ops each, `lost` records missing."""
    gen = torch.Generator("cuda").manual_seed(seed)
    rnd = lambda lo, hi, n: torch.randint(lo, hi, (n,), generator=gen, device="cuda")
    n_rec = sum(sizes) * n_seq
    i = torch.randperm(n_rec, generator=gen, device="cuda")[lost:]
    if order == "rank":
        i = torch.sort(i).values
    rank, seq, n = i // n_seq, i % n_seq, len(i)
    comm = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.tensor(sizes, device="cuda"))[rank]
    te = 1_000_000_000 + seq * 5_000_000 + rnd(0, 40_000, n)
    return dict(rank=rank.int(), comm=comm.int(), seq=seq.int(), op=torch.zeros(n, dtype=torch.uint8, device="cuda"),
                bytes=torch.full((n,), 16 * MiB, device="cuda"), t_enter=te, t_exit=te + rnd(1_000_000, 1_200_000, n))


def device_analyzer(sizes):
    an, r0 = ccld.Analyzer(), 0
    for c, n in enumerate(sizes):
        an.comm_register(c, list(range(r0, r0 + n)), 0, 0)
        r0 += n
    return an


def test_a_large_slot_table_filled_during_the_range_pass():
    """27 M slots in two windows, the second one's table at no 16-byte boundary, on memory that holds the indices of windows that lost
    other records: what the waiting pass, which fills its table with a copy of its own, finds."""
    sizes = [8] * 1500 + [5] * 301
    first = [device_job(sizes, 1001, s, lost=4000) for s in (1, 2)]
    then = [device_job(sizes, 1001, s, lost=4000) for s in (3, 4)]
    an = device_analyzer(sizes)
    for wins in (first, then):
        for w, c in enumerate(wins):
            an.trace_upload(w, c)
        for _ in range(2):
            an.reset()
            an.analyze_window(0, 2, 10**13)
            got = [an.get_optable(w) for w in (0, 1)]
        if wins is first:
            del got
            for w in (0, 1):
                an.window_release(w)
    assert an.get_route_counts() == {"unwaited": 3, "redone": 0, "packed": 0, "filled_under_range": 3}
    waiting = device_analyzer(sizes)
    waiting.set_speculation(False)
    for w, c in enumerate(then):
        waiting.trace_upload(w, c)
    waiting.analyze_window(0, 2, 10**13)
    for w in (0, 1):
        want = waiting.get_optable(w)
        for k in want:
            same(got[w][k], want[k], k)
    assert waiting.get_route_counts()["unwaited"] == 0


def test_pinned_upload_beyond_what_a_kernel_reads():
    """More than 32 MB of pinned columns are copied column by column."""
    rng = np.random.default_rng(8)
    n_seq = 100_000
    reg, cols, n = job([8], n_seq, rng, spacing=2_000_000)
    an, o = make_pair(reg)
    assert o.upload(0, cols) == 0 and sum(v.nbytes for v in cols.values()) > 32 << 20
    an.trace_upload(0, {k: torch.from_numpy(v if v.itemsize == 1 else v.view("i%d" % v.itemsize)).pin_memory() for k, v in cols.items()})
    an.analyze_window(0, 1, 10**15)
    assert o.analyze(0, 1, 10**15) == 0
    compare_window(an, o, 0)
