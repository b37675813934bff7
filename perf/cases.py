"""The work this framework is used for, as timed cases: whole analyses of profiling windows.

A pass is one analysis through the public entry points: open a window on the records at hand,
run the calls, take the results.  The results stay on the device, owned by the window, until
the same session analyses its next window (which closes the one before).  Inputs come from the
package's own generator: a stretch of at most 2^19 records is simulated on the host and repeated
along the time axis on the device, with fresh correlation ids, collective sequence numbers, times
and a pace of its own per repetition, until the window holds the records asked for; record buffers
of all processes then arrive in shuffled order.  Which calls are made is the case's; the pace of
every repetition, the delivery order and the hashes are the seed's.

Paths
  hot     the seven calls on records that are resident on the device; every result column and
          table is returned
  report  the seven calls and all analyses built on them (device overlap, gap blame, roll-up,
          operator efficiency, critical path and their symbol tables)
  host    the seven calls on records in host memory; the result tables are read back
  lane    the gap scan of one stream through the call that allocates no device memory
"""
import math

import numpy as np
import torch

from paper_2609_40247_b200 import synth, ta

STRETCH = 1 << 19  # records simulated on the host; longer windows repeat the stretch
BUFFER = 4096      # records of one delivery buffer
MIN_GAP_NS = 500_000
MAX_RECORDS = 66_800_000
PATH_SYMBOLS = 16 * 4096  # (process, symbol) pairs of the largest family


def _hot(name, family, records, windows=1, ids="dense", order="buffers", align=16, defects=False,
         memory="torch", path="hot"):
    return {"name": name, "path": path, "family": family, "records": records, "windows": windows,
            "ids": ids, "order": order, "align": align, "defects": defects, "memory": memory}


def listed():
    return [
        # a look at a live process: a few thousand records, the calls' own latency is all there is
        _hot("live look 2k", "c0", 2_400),
        # one stream's gaps inside a serving process that may not allocate
        {"name": "lane gaps 64k", "path": "lane", "records": 65_536},
        # the smallest configured window: one process, two streams
        _hot("single process 60k", "c0", 60_000),
        # everything the analyzer can say about a short prefill window
        _hot("report prefill 250k", "c2", 250_000, path="report"),
        # a collector hands over a host buffer of one tensor-parallel decode window
        _hot("host decode 1M", "c1", 1_000_000, path="host"),
        # hashed ids and symbols, records that arrive in no order at an odd place of a ring buffer,
        # some of them damaged
        _hot("hashed ids ragged 1.2M", "c3", 1_234_567, ids="hashed", order="shuffled", align=8,
             defects=True),
        # eight ranks of tensor-parallel decode, the configured size
        _hot("decode 4M", "c1", 4_194_304),
        # everything about a long mixture-of-experts window
        _hot("report experts 8M", "c3", 8_000_000, path="report"),
        # prefill with operator trees to depth eight, the configured size
        _hot("prefill 16M", "c2", 16_777_216),
        # a fleet's windows of one collection round, analysed in one pass
        _hot("fleet 512 windows 33M", "mix", 33_554_432, windows=512),
        # the headline window: 16 ranks of expert-parallel decode, memory from the library's pool
        _hot("experts 66M", "c3", MAX_RECORDS, memory="library"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choices(("hot", "fleet", "report", "host", "lane"), (10, 3, 4, 2, 1))[0]
    if path == "lane":
        return {"path": "lane", "records": _log_uniform(rng, 1_000, ta.NOALLOC_MAX_RECORDS)}
    if path == "fleet":
        windows = _log_uniform(rng, 3, 512)
        # a decode step of all ranks is some 20 000 records; the longest window is one stretch
        records = _log_uniform(rng, 20_000 * windows, min(33_000_000, windows * STRETCH * 2 // 3))
        case = _hot("", "mix", records, windows=windows)
    else:
        lo, hi = {"hot": (1_500, 33_000_000), "report": (20_000, 8_000_000), "host": (50_000, 4_000_000)}[path]
        records = _log_uniform(rng, lo, hi)
        families = ["c0"] if records < 300_000 else []
        families += ["c2"] + (["c1", "c3"] if records >= 40_000 else [])
        case = _hot("", rng.choice(families), records, path=path)
    if path != "report":
        case["ids"] = "hashed" if rng.random() < 0.15 else "dense"
    case["order"] = "shuffled" if path != "fleet" and rng.random() < 0.2 else "buffers"
    case["align"] = 8 if rng.random() < 0.2 else 16
    case["defects"] = rng.random() < 0.25
    case["memory"] = "library" if rng.random() < 0.3 else "torch"
    del case["name"]
    return case


# ------------------------------------------------------------------------------ inputs


def _stretch(family, records, number, fixed_span=False):
    """One simulated stretch of about `records` records (exactly so many when the span is fixed):
    n x 5 int64 words on the device with times from 0, the extent in ns, and the (communicator,
    ranks) pairs.  Word 3 = pid | name << 32, word 4 = seq | stream << 32 | kind << 48."""
    p = synth.window_params(family, records, number)
    if fixed_span:
        p["span_ns"] = synth.SPAN_30S
        p["n_steps"] += 1  # more than asked for, the rest is cut off below
        if family == "c3":
            p["comm_offset"] = 16  # 16-rank communicators get ids of their own
    ev, _, _ = synth.generate_window(p, synth.T0_BASE, truth=False)
    words = torch.from_numpy(np.ascontiguousarray(ev).view(np.int64).reshape(-1, 5)).cuda()
    words[:, :2] -= synth.T0_BASE
    if fixed_span:
        words = _first_by_start(words, records)
    comms = []
    if p["mode"] == 1:
        comms = [(0x5EED0000 + p["comm_offset"] + s, p["n_pid"])
                 for s in range(min(p["colls_per_layer"], p["n_streams"]))]
    return words, int(words[:, 1].max()) + 1000, comms


def _first_by_start(words, k):
    """The k records that start first, in the order they came in."""
    return words[torch.sort(torch.sort(words[:, 0], stable=True).indices[:k]).values]


def _kind(words):
    return words[:, 4] >> 48


def _pace(count, g):
    """Time scale of each repetition in 1/1024: 1 to 1.25 (never below 1: order and nesting stay)."""
    return torch.randint(1024, 1281, (count,), device="cuda", generator=g)


def _one_window(case, g):
    """Records of one window, its end and the communicators."""
    n = case["records"]
    base, extent, comms = _stretch(case["family"], min(n, STRETCH), 1 + n % 1000)
    full = n // len(base)
    tiles = full + (n % len(base) > 0)
    kind = _kind(base)
    coll = kind == ta.KIND_COLL
    joins = (kind == ta.KIND_LAUNCH) | (kind == ta.KIND_KERNEL) | (kind == ta.KIND_MEMCPY)
    ids = joins * int(base[joins, 2].max())
    seqs = coll * (int((base[:, 4] & 0xFFFFFFFF)[coll].max()) + 1 if comms else 0)
    pace = _pace(tiles, g)
    begin = torch.cumsum(extent * pace >> 10, 0) - (extent * pace >> 10) + torch.arange(tiles, device="cuda")

    def repeat(part, ids, seqs, first, last):
        r = torch.arange(first, last, device="cuda").view(-1, 1)
        out = part.unsqueeze(0).repeat(last - first, 1, 1)
        for c in (0, 1):
            out[:, :, c] = (out[:, :, c] * pace[first:last].view(-1, 1) >> 10) + begin[first:last].view(-1, 1)
        out[:, :, 2] += ids * r
        out[:, :, 4] += seqs * r
        return out.view(-1, 5)

    words = repeat(base, ids, seqs, 0, full)
    if tiles > full:  # the window closes in the middle of the last repetition
        rest = torch.cat([base, ids.view(-1, 1), seqs.view(-1, 1)], 1)
        rest = _first_by_start(rest, n - full * len(base))
        words = torch.cat([words, repeat(rest[:, :5], rest[:, 5], rest[:, 6], full, tiles)])
    words[:, :2] += synth.T0_BASE
    end = int(words[:, 0].max()) + 1
    if case["defects"]:
        _damage(words)
    if case["order"] == "shuffled":
        words = words[torch.randperm(n, device="cuda", generator=g)]
    elif n >= 2 * BUFFER:
        whole = n // BUFFER
        at = torch.randperm(whole, device="cuda", generator=g)
        words = torch.cat([words[:whole * BUFFER].view(whole, BUFFER, 5)[at].view(-1, 5),
                           words[whole * BUFFER:]])
    return words, max(end, synth.T0_BASE + synth.SPAN_30S), comms


def _fleet(case, g):
    """Windows of the decode, prefill and experts families in turn, of different lengths."""
    W = case["windows"]
    k = min(W, 6)
    lengths = np.random.RandomState(W).uniform(0.6, 1.4, k) * case["records"] / W
    parts, comms = [], {}
    for j in range(k):
        words, _, c = _stretch(("c1", "c2", "c3")[j % 3], int(lengths[j]), 1 + j, fixed_span=True)
        parts.append(words)
        comms.update(c)
    sizes = np.array([len(parts[w % k]) for w in range(W)])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    words = torch.cat([torch.cat(parts).repeat(W // k, 1)] + parts[:W % k])
    window = torch.repeat_interleave(torch.arange(W, device="cuda"), torch.from_numpy(sizes).cuda())
    pace = _pace(W, g)[window]
    for c in (0, 1):
        words[:, c] = (words[:, c] * pace >> 10) + (synth.T0_BASE + window * synth.WINDOW_STRIDE_NS)
    if case["defects"]:
        _damage(words)
    t0 = synth.T0_BASE + np.arange(W, dtype=np.int64) * synth.WINDOW_STRIDE_NS
    return words, off, t0, t0 + synth.SPAN_30S, sorted(comms.items())


def _hash_ids(words, seed):
    """Correlation ids as hashes of 62 bits and symbols as hashes of 31 bits."""
    coll = _kind(words) == ta.KIND_COLL
    mixed = ((words[:, 2] + seed) * -7046029254386353131) & 0x3FFFFFFFFFFFFFFF
    words[:, 2] = torch.where(coll, words[:, 2], mixed)
    name = ((words[:, 3] >> 32) * 2654435761) & 0x7FFFFFFF
    words[:, 3] = (words[:, 3] & 0xFFFFFFFF) | (name << 32)


def _damage(words):
    """Three records in a thousand are unusable: unknown kind, end before start, outside the window."""
    m = len(words)
    for what in range(3):
        at = torch.arange(37 + what, m, 1000, device="cuda")
        if what == 0:
            words[at, 4] = (words[at, 4] & 0x0000FFFFFFFFFFFF) | (9 << 48)
        elif what == 1:
            words[at, 1] = words[at, 0] - 5
        else:
            words[at, 0] = synth.T0_BASE - 1_000


def _op_work(words, g):
    """Operation count and data volume per input record, as synth.op_work gives them."""
    m = len(words)
    name = words[:, 3] >> 32
    batch = torch.randint(1, 65, (m,), device="cuda", generator=g).double()
    hidden = (1024 * (1 + name % 8)).double()
    gemm = name % 3 != 0
    known = (_kind(words) == ta.KIND_OP) & (torch.rand(m, device="cuda", generator=g) >= 0.03)
    flops = torch.where(gemm, 2.0 * batch * hidden * hidden, 4.0 * batch * hidden)
    nbytes = torch.where(gemm, 2.0 * (hidden * hidden + 2.0 * batch * hidden), 6.0 * batch * hidden)
    return torch.where(known, flops, -1.0).contiguous(), torch.where(known, nbytes, -1.0).contiguous()


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n = case["records"]
    if case["path"] == "lane":
        dur = torch.empty(n, device="cuda", dtype=torch.float64).log_normal_(math.log(4000.0), 1.2, generator=g)
        idle = torch.empty(n, device="cuda", dtype=torch.float64).exponential_(1.0 / 3000.0, generator=g)
        idle *= torch.rand(n, device="cuda", generator=g) < 0.5  # back to back as often as not
        dur, idle = dur.long().clamp_(min=500), idle.long()
        end = synth.T0_BASE + torch.cumsum(dur + idle, 0)
        return {"case": case, "ts_start": (end - dur).contiguous(), "ts_end": end,
                "t0": synth.T0_BASE, "t1": max(int(end[-1]) + 1, synth.T0_BASE + synth.SPAN_30S),
                "gap_before": torch.empty(n, dtype=torch.int64, device="cuda"),
                "lane_out": torch.empty(ta.LANE_GAPS.itemsize, dtype=torch.uint8, device="cuda")}
    if case["windows"] > 1:
        words, off, t0, t1, comms = _fleet(case, g)
    else:
        words, end, comms = _one_window(case, g)
        off = np.array([0, len(words)], dtype=np.int64)
        t0, t1 = np.array([synth.T0_BASE], dtype=np.int64), np.array([end], dtype=np.int64)
    if case["ids"] == "hashed":
        _hash_ids(words, seed)
    if case["align"] == 8:  # the records begin at an odd record of a larger buffer
        room = torch.empty((len(words) + 1, 5), dtype=torch.int64, device="cuda")
        room[1:] = words
        words = room[1:]
    st = {"case": case, "off": off, "t0": t0, "t1": t1, "comms": comms, "window": None}
    if case["path"] == "report":
        st["flops"], st["nbytes"] = _op_work(words, g)
    if case["path"] == "host":
        st["events"] = words.cpu().numpy().reshape(-1).view(ta.EVENT_DTYPE)
        st["long_gaps"] = np.zeros(len(words) // 8 + 64, dtype=ta.LONG_GAP)
    else:
        st["events"] = words.contiguous()
        # the session's own lists where the times decide how long a list is: the long gaps, and
        # the symbols the critical paths run through
        room = len(words) // 8 + 64
        st["long_gaps"] = torch.zeros(room * ta.LONG_GAP.itemsize, dtype=torch.uint8, device="cuda")
        st["b_class"] = torch.full((room,), -1, dtype=torch.int32, device="cuda")
        st["b_launch"] = torch.full((room,), -1, dtype=torch.int32, device="cuda")
        if case["path"] == "report":
            for k, dt in _AGG.items():
                rows = PATH_SYMBOLS * (ta.NBINS if k == "g_hist" else 1)
                st[k] = torch.full((rows,), -1, dtype=dt, device="cuda")
    return st


# -------------------------------------------------------------------------------- passes

_SORT = {"perm": torch.int32, "ts_start": torch.int64, "ts_end": torch.int64, "corr_id": torch.int64,
         "pid": torch.int32, "name_id": torch.int32, "seq": torch.int32, "stream": torch.int16,
         "kind": torch.int16, "lane_window": torch.int32, "lane_pid": torch.int32,
         "lane_stream": torch.int16, "lane_domain": torch.int16, "lane_off": torch.int32}
_JOIN = {"launch_of": torch.int32, "launch_latency": torch.int64, "queue_delay": torch.int64,
         "kernels_of_launch": torch.int32}
_ATTR = {"parent": torch.int32, "depth": torch.uint8, "op_of": torch.int32, "op_first_start": torch.int64,
         "op_last_end": torch.int64, "op_kernel_ns": torch.int64, "op_n_kernels": torch.int32}
_GAPS = {"gap_before": torch.int64, "lane_gaps": torch.int64, "lane_hist": torch.int32,
         "win_hist": torch.int32}
_AGG = {"g_window": torch.int32, "g_pid": torch.int32, "g_name": torch.int32, "g_count": torch.int64,
        "g_sum": torch.int64, "g_min": torch.int64, "g_max": torch.int64, "g_hist": torch.int32}
_COLL = {"g_window": torch.int32, "g_comm": torch.int64, "g_seq": torch.int32, "g_n_members": torch.int32,
         "g_min_start": torch.int64, "g_max_start": torch.int64, "g_skew": torch.int64,
         "g_max_end": torch.int64, "g_straggler_pid": torch.int32, "g_flags": torch.int32,
         "wait_ns": torch.int64, "r_window": torch.int32, "r_pid": torch.int32, "r_n_coll": torch.int64,
         "r_sum_wait": torch.int64, "r_max_wait": torch.int64, "r_n_straggler": torch.int64}
_ROLL = {"incl_n_kernels": torch.int32, "incl_first_start": torch.int64, "incl_last_end": torch.int64,
         "incl_kernel_ns": torch.int64, "replay_first_start": torch.int64, "replay_last_end": torch.int64,
         "replay_kernel_ns": torch.int64}
_OVER = {"d_window": torch.int32, "d_pid": torch.int32, "d_n_events": torch.int64, "d_busy": torch.int64,
         "d_idle": torch.int64, "d_compute": torch.int64, "d_comm": torch.int64, "d_overlap": torch.int64,
         "d_exposed": torch.int64}
_SOL = {"sol_mfu": torch.float64, "sol_mbu": torch.float64, "sol_op": torch.float64, "sol_state": torch.uint8}
_PATH = {"on_path": torch.uint8, "cp_window": torch.int32, "cp_pid": torch.int32, "cp_sink": torch.int32,
         "cp_n_nodes": torch.int32, "cp_reason": torch.int32, "cp_begin": torch.int64,
         "cp_end": torch.int64, "cp_ns": torch.int64}


def _columns(result, names):
    return [result.tensor(k).view(dt) for k, dt in names.items()]


def _keep(st, key, rows):
    """Puts a list whose length depends on the times at the front of the session's own buffer."""
    st[key][:len(rows)] = rows
    return st[key]


def _words(summary):
    return summary.view(np.int64).reshape(-1)


def run(st):
    case = st["case"]
    if case["path"] == "lane":
        gap, lane = ta.lane_gaps_noalloc(st["ts_start"], st["ts_end"], st["t0"], st["t1"],
                                         st["gap_before"], st["lane_out"])
        return [gap, [int(lane[k]) for k in ta.LANE_GAPS.names]]
    if st["window"] is not None:
        st["window"].close()
    w = st["window"] = ta.Window(st["events"], st["off"], st["t0"], st["t1"],
                                 use_torch_allocator=case["memory"] == "torch")
    s = w.sort_timeline()
    j = w.correlate_launches()
    a = w.attribute_operators()
    gaps = w.stream_gaps(MIN_GAP_NS)
    k1 = w.aggregate_ops(ta.DEVICE_KINDS, 0)
    k2 = w.aggregate_ops(1 << ta.KIND_OP, 1)
    c = w.match_collectives(st["comms"])
    found = np.concatenate([_words(w.load_summary), _words(j.join_sum), _words(a.attr_sum)])
    if case["path"] == "host":
        out = [found]
        for result, names in ((s, ("lane_window", "lane_pid", "lane_stream", "lane_domain", "lane_off")),
                              (gaps, ("lane_hist", "win_hist")), (k1, _AGG), (k2, _AGG),
                              (c, [k for k in _COLL if k != "wait_ns"])):
            out += [result.numpy(k) for k in names]
        return out + [_words(gaps.numpy("lane_gaps")), _words(_keep(st, "long_gaps", gaps.numpy("long_gaps")))]
    listed_gaps = _keep(st, "long_gaps", gaps.tensor("long_gaps"))
    if case["path"] == "hot":
        return [found, listed_gaps] + _columns(s, _SORT) + _columns(j, _JOIN) + _columns(a, _ATTR) + \
            _columns(gaps, _GAPS) + _columns(k1, _AGG) + _columns(k2, _AGG) + _columns(c, _COLL)
    o = w.device_overlap()
    b = w.blame_gaps(gaps)
    k3 = w.aggregate_ops(1 << ta.KIND_OP, 2)
    r = w.rollup_operators()
    f = w.operator_sol(st["flops"], st["nbytes"], synth.PEAK_FLOPS, synth.PEAK_BW)
    p = w.critical_path()
    k4 = w.aggregate_ops(62, 3)
    # of the seven calls, what the analyses are read against; "hot" returns all of it
    sol = f.sol_sum
    return [found, _words(r.rollup_sum), _words(b.blame_sum), _words(p.critpath_sum),
            _words(sol)[:4], sol["sum_flops"], sol["sum_bytes"], sol["max_sol"],
            s.tensor("perm").view(torch.int32), s.tensor("lane_off").view(torch.int32),
            j.tensor("launch_of").view(torch.int32), a.tensor("op_of").view(torch.int32), listed_gaps,
            _keep(st, "b_class", b.tensor("b_class").view(torch.int32)),
            _keep(st, "b_launch", b.tensor("b_launch").view(torch.int32)),
            b.tensor("op_gap_ns").view(torch.int64)] + \
        _columns(o, _OVER) + _columns(k3, _AGG) + _columns(r, _ROLL) + _columns(f, _SOL) + \
        _columns(p, _PATH) + [_keep(st, k, k4.tensor(k).view(dt)) for k, dt in _AGG.items()]


# ----------------------------------------------------------------------------------- bounds


def work(case):
    """Each input byte read once, each result column written once; every value is an integer, so
    there is no arithmetic to speak of."""
    n = case["records"]
    if case["path"] == "lane":
        return {"bytes": 24.0 * n, "flops": 0.0}
    # records 40; out: sorted columns and permutation 44, join 24, attribution 37, gaps 8, waits 8
    per = 40 + 44 + 24 + 37 + 8 + 8
    if case["path"] == "report":
        per += 16 + 52 + 8 + 25 + 1  # counts in; out: roll-up, idle charged, efficiency, path marks
    return {"bytes": float(per) * n, "flops": 0.0}


def tolerance(case):
    # the sums of operation counts (32-bit-sized terms in doubles, any order): n * 2^-53 for the
    # 10^7 terms of the largest window; everything else is whole numbers or single quotients
    return {"rel": 1e-9, "max": 1e-9, "differ": 0.0} if case["path"] == "report" else "exact"
