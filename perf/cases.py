"""The work a user has the analyzer do, as measurable cases.

A case is a dict of plain values. `prepare` makes what the user's program holds before the call - trace columns, an
Analyzer with its communicators registered - from a seed alone; `run` is one pass through the public entry points;
`work` is what a pass cannot do without; `tolerance` is how far another correct implementation may be off.

Four kinds of pass:
  monitor   the analyzer service: a window's columns arrive in host memory, are uploaded, analysed, the verdict and
            the rank statistics are read and the window is dropped (one window per minute and job, the deployed use)
  analyze   windows that already sit in device memory (a collector that writes to the GPU, or a backlog): analysed as one
            batch, every window's verdict and the cumulative rank statistics read, the per-op tables taken as device arrays
  rates     SendCount / RecvCount changes per op from the raw samples of the rank probes, the step before a window is uploaded
  diagnose  the questions asked about an analysed window: hang location for every alert and by name, op-set
            consistency, per-op table, ranges and rank statistics on the host

and four kinds of job:
  3d        TP x PP x DP training: rings of `tp`, `pp` and `dp` ranks, five op slots TP TP PP TP DP per repetition
  world     one communicator of `dp` ranks
  stress    node-local rings of 8, blocks of `pp` ranks, one ring across the nodes per local rank (`dp` nodes), and a ring
            over half the nodes that hangs at its last op
  rings     `pp` rings (or trees) of `dp` ranks; the last op of one of them hangs

Times are drawn like the traces of such jobs: ops 5 ms apart, arrival jitter N(0, 20 us), durations lognormal around 2 ms
per 16 MiB, message sizes lognormal around 32 MiB, one rank in a thousand late (exponential, 500 us mean, on a fifth of its
ops) and one in a thousand on a link of half the bandwidth. `lost` records per million never arrive.
"""
import math

import numpy as np
import torch

import paper_2605_04478_b200 as ccld

ALLREDUCE, ALLGATHER, REDUCESCATTER, SENDRECV = 0, 1, 2, 4
MS = 1_000_000
SPACING = 5 * MS
T0 = 1000 * MS
COUNTS = ("n_records", "n_groups", "n_slots", "n_rejected", "n_complete", "n_incomplete", "n_barrier", "n_analysed", "n_flag_skew",
          "n_flag_dur", "n_opset_mismatch", "error_bits", "n_comm_rows_total", "n_alerts_total", "n_suspects_total", "rc")
HANG = ("cls", "n_roots_total", "n_not_entered", "n_hung", "n_not_hung", "n_missing_frames", "stuck_step", "n_members", "min_total")
OPSET = ("n_members", "n_present", "n_deviating_total", "majority_count", "op", "algo", "proto", "bytes")


def listed():
    return [
        # the smallest job that is watched: one node, one ring, a window of 1,000 AllReduces in pageable host memory
        dict(name="monitor_8", kind="monitor", job="3d", tp=8, pp=1, dp=1, reps=333, lost=0, pinned=False, rates=True),
        # an ordinary job: 512 ranks, 1,000 ops per rank, columns in pinned host memory, a few records lost on the way
        dict(name="monitor_512", kind="monitor", job="3d", tp=8, pp=8, dp=8, reps=200, lost=20, pinned=True, rates=True),
        # the same job with 3,000 ops per rank and window, columns on the device
        dict(name="window_512", kind="analyze", job="3d", tp=8, pp=8, dp=8, reps=600, windows=1, lost=0, order="rank", rates=True),
        # the large job: 4,096 ranks, a backlog of twelve windows of 1,000 ops per rank (49 M records)
        dict(name="backlog_4096", kind="analyze", job="3d", tp=8, pp=8, dp=64, reps=200, windows=12, lost=0, order="rank", rates=True),
        # records in the order in which the probes reported them
        dict(name="arrival_4096", kind="analyze", job="3d", tp=8, pp=8, dp=64, reps=200, windows=2, lost=0, order="arrival", rates=True),
        # no power of two anywhere: 4 x 6 x 172 ranks, odd op counts, lost records, probes without the rate columns
        dict(name="ragged_4128", kind="analyze", job="3d", tp=4, pp=6, dp=172, reps=117, windows=2, lost=50, order="rank", rates=False),
        # pure data parallelism: one communicator of 4,096 ranks
        dict(name="world_4096", kind="analyze", job="world", tp=1, pp=1, dp=4096, reps=1000, windows=2, lost=0, order="rank", rates=True),
        # the largest job: 16,384 ranks, rings of 8 to 2,048, a ring of 1,024 that hangs, progress frames uploaded with it
        dict(name="stress_16384", kind="analyze", job="stress", tp=8, pp=128, dp=2048, reps=10, windows=1, lost=0, order="rank", rates=True),
        # the hang case: sixteen rings of 256, a hundred completed AllReduces and one that never completes
        dict(name="hang_4096", kind="analyze", job="rings", tp=1, pp=16, dp=256, reps=101, windows=1, lost=0, order="rank", rates=True),
        # what is asked once an alert is up, on trees of 1,024 ranks
        dict(name="diagnose_1024", kind="diagnose", job="rings", tp=1, pp=4, dp=1024, reps=50, tree=True, lost=0, rates=True),
        # probe samples of one window of the large job: 4,096 ranks, 1,000 ops each, one sample per millisecond
        dict(name="rates_4096", kind="rates", ranks=4096, ops=1000),
        # and of one node
        dict(name="rates_8", kind="rates", ranks=8, ops=999),
    ]


def _span(rng, lo, hi):
    """Whole numbers of [lo, hi], evenly over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(("monitor", "monitor", "analyze", "analyze", "analyze", "analyze", "diagnose", "rates"))
    if kind == "rates":
        ranks = _span(rng, 8, 8192)
        return dict(kind="rates", ranks=ranks, ops=_span(rng, 20, min(3000, 6_000_000 // ranks)))
    if kind == "diagnose":
        n = _span(rng, 4, 4096)
        return dict(kind=kind, job="rings", tp=1, pp=_span(rng, 1, max(1, 8192 // n)), dp=n, reps=_span(rng, 2, 60), tree=rng.random() < 0.5,
                    lost=0, rates=True)
    job = "3d" if kind == "monitor" else rng.choice(("3d", "3d", "3d", "world", "stress", "rings"))
    case = dict(kind=kind, job=job, lost=rng.choice((0, 0, 20, 100)), rates=rng.random() < 0.8)
    most = 3_000_000 if kind == "monitor" else 16_000_000          # records per window
    if job == "3d":
        case.update(tp=rng.choice((2, 4, 8, 8, 8)), pp=rng.choice((1, 2, 3, 4, 6, 8)))
        case["dp"] = _span(rng, 1, min(1500, most // (case["tp"] * case["pp"] * 15)))
        case["reps"] = _span(rng, 3, max(3, min(700, most // (case["tp"] * case["pp"] * case["dp"] * 5))))
    elif job == "world":
        case.update(tp=1, pp=1, dp=_span(rng, 9, 8192))
        case["reps"] = _span(rng, 5, max(5, min(3000, most // case["dp"])))
    elif job == "stress":
        nodes = 32 * _span(rng, 4, 64)
        case.update(tp=8, pp=rng.choice((64, 128, 256)), dp=nodes, reps=_span(rng, 1, max(1, min(10, most // (nodes * 808)))), lost=0)
    else:
        case.update(tp=1, pp=_span(rng, 1, 32), dp=_span(rng, 5, 1500), lost=0)
        case["reps"] = _span(rng, 3, max(3, min(700, most // (case["pp"] * case["dp"]))))
    if kind == "monitor":
        case["pinned"] = rng.random() < 0.5
    else:
        case["order"] = rng.choice(("rank", "rank", "rank", "arrival"))
        per = _records(case)
        case["windows"] = _span(rng, 1, max(1, min(12, (40_000_000 if case["order"] == "rank" else 8_000_000) // per)))
        if job in ("stress", "rings"):
            case["windows"] = 1                                     # the hang ends the trace
    return case


# ---- jobs -----------------------------------------------------------------------------------------------------------

def _strided(ranks, n, stride):
    """Groups {first + i * stride, i < n} that tile [0, ranks), as a [ranks / n, n] array."""
    r = np.arange(ranks, dtype=np.int64)
    return r[(r % (n * stride)) < stride][:, None] + np.arange(n, dtype=np.int64)[None, :] * stride


def _families(case):
    """[(members [groups, n] in ring order, op codes in turn)], the family of each op slot, whether the last family's first group hangs."""
    tp, pp, dp = case["tp"], case["pp"], case["dp"]
    if case["job"] == "3d":
        R = tp * pp * dp
        fams = [(_strided(R, tp, 1), (ALLREDUCE,)), (_strided(R, pp, tp), (SENDRECV,)), (_strided(R, dp, tp * pp), (REDUCESCATTER, ALLGATHER))]
        keep = [k for k, n in enumerate((tp, pp, dp)) if n > 1]
        return [fams[k] for k in keep], [keep.index(k) for k in (0, 0, 1, 0, 2) if k in keep], False
    if case["job"] == "world":
        return [(_strided(dp, dp, 1), (ALLREDUCE,))], [0], False
    if case["job"] == "stress":
        R = 8 * dp
        ring = (np.arange(dp // 2, dtype=np.int64) * 8 + 3)[None, :]
        return [(_strided(R, 8, 1), (ALLREDUCE,)), (_strided(R, pp, 1), (ALLGATHER, REDUCESCATTER)), (_strided(R, dp, 8), (ALLREDUCE,)),
                (ring, (ALLREDUCE,))], [0, 0, 1, 2] * 25 + [3], True
    return [(_strided(pp * dp, dp, 1), (ALLREDUCE,))], [0], True


def _sizes(case):
    """Records, groups, slots, communicators and ranks of a window (without losses)."""
    fams, pat, _ = _families(case)
    ops = [pat.count(f) * case["reps"] for f in range(len(fams))]
    rec = sum(m.size * k for (m, _), k in zip(fams, ops))
    return rec, sum(m.shape[0] * k for (m, _), k in zip(fams, ops)), sum(m.shape[0] for m, _ in fams), 1 + max(int(m.max()) for m, _ in fams)


def _records(case):
    return _sizes(case)[0]


def _window(case, w, gen, dev):
    """Columns of window w on `dev`, its progress frames (or None) and the analyzer's clock after it."""
    fams, pat, hangs = _families(case)
    L, O = len(pat), len(pat) * case["reps"]
    R = 1 + max(int(m.max()) for m, _ in fams)
    rnd = lambda *s: torch.rand(*s, generator=gen, device=dev)
    nrm = lambda *s: torch.randn(*s, generator=gen, device=dev)
    pat_t = torch.tensor(pat, device=dev)
    occ = torch.tensor([pat[:i].count(pat[i]) for i in range(L)], device=dev)
    cnt = torch.tensor([pat.count(f) for f in range(len(fams))], device=dev)
    o = torch.arange(O, device=dev)
    fam_o = pat_t[o % L]
    seq_o = (o // L) * cnt[fam_o] + occ[o % L]                       # op counter inside the window; windows follow each other
    comm = torch.full((R, O), -1, dtype=torch.int64, device=dev)
    op = torch.zeros((R, O), dtype=torch.uint8, device=dev)
    size = torch.zeros((R, O), dtype=torch.int64, device=dev)
    c0 = 0
    for f, (members, codes) in enumerate(fams):
        at = (fam_o == f).nonzero().flatten()
        m = torch.from_numpy(members).to(dev)
        G = m.shape[0]
        grp = torch.full((R,), -1, dtype=torch.int64, device=dev)
        grp[m.reshape(-1)] = torch.arange(G, device=dev).unsqueeze(1).expand_as(m).reshape(-1)
        b = ((32 << 20) * torch.exp(nrm(G, at.numel()))).clamp(4 << 10, 4 << 30).to(torch.int64) & ~3     # one size per op, the same on all ranks
        size[:, at] = b[grp.clamp(min=0)]
        comm[:, at] = torch.where(grp >= 0, grp + c0, -1).unsqueeze(1).expand(R, at.numel())
        op[:, at] = torch.tensor(codes, dtype=torch.uint8, device=dev)[seq_o[at] % len(codes)].unsqueeze(0).expand(R, -1)
        c0 += G
    late = rnd(R, 1) < 0.001
    slow = rnd(R, 1) < 0.001
    t_enter = T0 + (w * O + o).unsqueeze(0) * SPACING + (20_000 * nrm(R, O)).to(torch.int64)
    t_enter += torch.where(late & (rnd(R, O) < 0.2), (-500_000 * torch.log(rnd(R, O).clamp(min=1e-6))).to(torch.int64), 0)
    dur = ((size >> 3).to(torch.float32) * torch.exp(0.1 * nrm(R, O)) * torch.where(slow, 2.0, 1.0)).to(torch.int64).clamp(min=1)
    t_exit = t_enter + dur
    chg = ((dur + MS - 1) // MS).to(torch.int32)
    seq = (w * case["reps"] * cnt[fam_o] + seq_o).to(torch.int32).unsqueeze(0).expand(R, O)
    frames, channels = None, 0
    if hangs:                                                        # the last op of the last family's first group never completes
        f = len(fams) - 1
        G, n = fams[f][0].shape
        ring0, last, channels = c0 - G, int(cnt[f]) * case["reps"] - 1, 8
        t_exit = torch.where((comm == ring0) & (seq == last), -1, t_exit)
        prog = torch.full((G, n, channels, 2), 64, dtype=torch.int32, device=dev)
        stuck = int(torch.randint(n, (1,), generator=gen, device=dev))
        prog[0] = 42
        prog[0, stuck] = 41
        frames = {"f_rank": torch.from_numpy(fams[f][0].reshape(-1).astype(np.int32)).to(dev),
                  "f_comm": torch.arange(ring0, c0, dtype=torch.int32, device=dev).repeat_interleave(n),
                  "f_seq": torch.full((G * n,), last, dtype=torch.int32, device=dev), "progress": prog.reshape(G * n, channels, 2)}
    keep = comm >= 0
    if case["lost"]:
        keep &= rnd(R, O) >= case["lost"] * 1e-6
    at = keep.reshape(-1).nonzero().flatten()
    if case.get("order", "rank") == "arrival":
        end = t_exit.reshape(-1)[at]
        at = at[torch.argsort(torch.where(end < 0, 1 << 62, end), stable=True)]
    pick = lambda t: t.reshape(-1)[at]
    cols = {"rank": (at // O).to(torch.int32), "comm": pick(comm).to(torch.int32), "seq": pick(seq), "op": pick(op), "bytes": pick(size),
            "t_enter": pick(t_enter), "t_exit": pick(t_exit)}
    if case["rates"]:
        cols["send_chg"] = pick(chg)
        cols["recv_chg"] = pick(chg + (rnd(R, O) < 0.1).to(torch.int32))
    return cols, frames, channels, T0 + (w + 1) * O * SPACING + 600_000 * MS


def _samples(case, gen, dev):
    """Records of one window and the probe samples (one per millisecond, every rank with its own phase and sample count) behind them."""
    R, O = case["ranks"], case["ops"]
    enter = T0 + torch.arange(O, device=dev).unsqueeze(0) * SPACING + (20_000 * torch.randn(R, O, generator=gen, device=dev)).to(torch.int64)
    dur = (4 * MS * torch.exp(torch.randn(R, O, generator=gen, device=dev))).clamp(max=500 * MS).to(torch.int64)
    exit_ = enter + dur
    exit_[:, -1] = torch.where(torch.rand(R, generator=gen, device=dev) < 0.01, -1, exit_[:, -1])
    T = O * SPACING // MS + 600
    n = T - torch.randint(0, 5, (R,), generator=gen, device=dev)
    n = torch.where(torch.rand(R, generator=gen, device=dev) < 0.005, n // 2, n)              # a probe that was restarted
    tick = (T0 - 10 * MS + torch.randint(0, MS, (R, 1), generator=gen, device=dev)) + torch.arange(T, device=dev).unsqueeze(0) * MS
    keep = torch.arange(T, device=dev).unsqueeze(0) < n.unsqueeze(1)
    step = lambda p: torch.cumsum((torch.rand(R, T, generator=gen, device=dev) < p).to(torch.int32), dim=1, dtype=torch.int32)[keep]
    off = torch.zeros(R + 1, dtype=torch.int64, device=dev)
    off[1:] = torch.cumsum(n, 0)
    rank = torch.arange(R, dtype=torch.int32, device=dev).unsqueeze(1).expand(R, O).reshape(-1).contiguous()
    return [rank, enter.reshape(-1), exit_.reshape(-1), off, tick[keep], step(0.7), step(0.6)]


# ---- the four functions a measurement calls --------------------------------------------------------------------------

def _analyzer(case):
    an = ccld.Analyzer()
    cid = 0
    for members, _ in _families(case)[0]:
        n = members.shape[1]
        for row in members:
            an.comm_register(cid, row, 1 if case.get("tree") else 0, 0)
            if case.get("tree"):
                an.comm_set_layers(cid, [int(math.log2(p + 1)) for p in range(n)])            # a binary tree in heap order
            cid += 1
    return an


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(dev).manual_seed(seed)
    if case["kind"] == "rates":
        return dict(kind="rates", an=ccld.Analyzer(), cols=_samples(case, gen, dev))
    an = _analyzer(case)
    state = dict(kind=case["kind"], an=an, ranks=_sizes(case)[3], windows=case.get("windows", 1), frames=None, channels=0)
    if case["kind"] == "monitor":
        cols, _, _, state["now"] = _window(case, 0, gen, dev)
        cols = {k: v.cpu() for k, v in cols.items()}
        state["cols"] = {k: v.pin_memory() if case["pinned"] else v.numpy() for k, v in cols.items()}
        state["next"] = 0
        return state
    for w in range(state["windows"]):
        cols, frames, channels, state["now"] = _window(case, w, gen, dev)
        an.trace_upload(w, cols, frames, channels)                    # borrowed: no copy
        if case["kind"] == "diagnose":                                # the codes of the Operation Type Set, one rank in fifty on another protocol
            n = cols["rank"].numel()
            proto = (torch.rand(state["ranks"], generator=gen, device=dev) < 0.02).to(torch.uint8)[cols["rank"].long()]
            an.trace_attach_opset(w, torch.zeros(n, dtype=torch.uint8, device=dev), proto)
    if case["kind"] == "diagnose":
        an.analyze_window(0, 1, state["now"])
        al = an.get_verdict(0)["alerts"]
        state["alert"] = (int(al["comm"][0]), int(al["seq"][0]))
        state["checks"] = [(c, case["reps"] // 2) for c in range(min(4, case["pp"]))]
    return state


class _View:
    """A device array of the library as PyTorch takes it without a copy; keeps the analyzer that owns the memory."""

    def __init__(self, owner, ptr, n, kind):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": kind, "data": (ptr, False), "version": 2}


def _table(an, w):
    """The per-op table of a window as device tensors."""
    t = an.get_optable(w, to_host=False)
    take = lambda names, n, kind: {k: torch.as_tensor(_View(an, t[k], n, kind), device="cuda") for k in names}
    G, S = t["n_groups"], t["n_slots"]
    return {**take(ccld.OPTABLE_I64, G, "<i8"), **take(ccld.OPTABLE_U32, G, "<i4"), **take(("busbw",), G, "<f8"), **take(("flags",), S, "|u1"),
            **take(("perm",), S, "<i4")}


def _counts(vs):
    return np.array([[v[k] for k in COUNTS] for v in vs], dtype=np.int64)


def _full(a, n):
    """A list of up to n entries as an array of n: the caller's table, of the same size whatever the trace holds."""
    out = np.zeros(n, a.dtype)
    out[:len(a)] = a
    return out


def _suspects(v, ranks):
    return {k: _full(a, 2 * ranks) for k, a in v["suspects"].items()}


def _hangs(hs):
    """Verdicts of the decision tree as one array, and their root lists (64 roots each at most)."""
    return np.array([[h[k] for k in HANG] for h in hs], dtype=np.int64), np.array([_full(h["roots"][:64], 64) for h in hs])


def run(state):
    an = state["an"]
    if state["kind"] == "rates":
        return an.derive_rates(*state["cols"])
    if state["kind"] == "monitor":
        w = state["next"]
        state["next"] = w + 1
        an.trace_upload(w, state["cols"])
        an.analyze_window(w, 1, state["now"])
        v = an.get_verdict(w)
        stats = an.get_rank_stats(state["ranks"])
        an.window_release(w)
        return {"counts": _counts([v]), "stats": stats, "rows": v["comm_rows"], "alerts": v["alerts"], "suspects": _suspects(v, state["ranks"])}
    if state["kind"] == "diagnose":
        c, s = state["alert"]
        checks = [an.opset_check(0, *x) for x in state["checks"]]
        table = an.get_optable(0)
        return {"sweep": _hangs(an.locate_hangs(0)), "asked": _hangs([an.locate_hang(0, c, s)]),
                "opset": np.array([[x[k] for k in OPSET] for x in checks], dtype=np.int64), "deviating": [_full(x["ranks"], state["ranks"]) for x in checks],
                "ranges": an.get_ranges(0), "stats": an.get_rank_stats(state["ranks"]),
                **{"op_" + k: table[k] for k in table}}
    W = state["windows"]
    an.reset()
    an.analyze_window(0, W, state["now"])
    vs = [an.get_verdict(w) for w in range(W)]
    out = {"counts": _counts(vs), "suspects": _suspects(vs[-1], state["ranks"]), "stats": an.get_rank_stats(state["ranks"]),
           "rows": {k: np.concatenate([v["comm_rows"][k] for v in vs]) for k in vs[0]["comm_rows"]}}
    if vs[-1]["n_alerts_total"]:
        out["alerts"] = vs[-1]["alerts"]
        out["hangs"] = _hangs(an.locate_hangs(W - 1))
    out["table"] = _table(an, W - 1)
    if W > 1:
        out["flags"] = [_only_flags(an, w) for w in range(W - 1)]
    return out


def _only_flags(an, w):
    t = an.get_optable(w, to_host=False)
    return torch.as_tensor(_View(an, t["flags"], t["n_slots"], "|u1"), device="cuda")


def work(case):
    """Each input column read once; each record's flag and record index, each op's row and each communicator's row written once."""
    if case["kind"] == "rates":
        ticks = case["ranks"] * (case["ops"] * SPACING // MS + 598)
        return {"bytes": 16 * ticks + 28 * case["ranks"] * case["ops"], "flops": 0}
    rec, groups, comms, ranks = _sizes(case)
    if case["kind"] == "diagnose":                                    # columns of the asked ops, the table and the statistics out
        return {"bytes": 5 * rec + 104 * groups + 40 * comms + 36 * ranks + (min(4, case["pp"]) + 2) * case["dp"] * 80, "flops": 0}
    per_window = (45 if case["rates"] else 37) * rec + 5 * rec + 104 * groups + 112 * comms
    return {"bytes": case.get("windows", 1) * per_window, "flops": 0}


def tolerance(case):
    """Whole numbers and flags are exact. Bandwidths, R and P are 64-bit quotients, and sums of up to some 10,000 of them in any order."""
    return "exact" if case["kind"] == "rates" else {"rel": 1e-12}
