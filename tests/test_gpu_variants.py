"""The two sides of each rule that chooses a way by sizes, value ranges or lanes, at the sizes where
they can go wrong, bit for bit against the oracle."""
import numpy as np
import pytest

from helpers import make_events
from paper_2609_40247_b200.synth import EVENT_DTYPE
from test_gpu_parity import both

pytestmark = pytest.mark.gpu

T0 = 1_700_000_000_000_000_000


def _device(n, starts, durations, pid=0, stream=0, kind=3, name=0):
    ev = np.zeros(n, dtype=EVENT_DTYPE)
    ev["ts_start"], ev["ts_end"] = starts, starts + durations
    ev["pid"], ev["stream"], ev["kind"], ev["name_id"] = pid, stream, kind, name
    ev["corr_id"] = -1 - np.arange(n)
    return ev


@pytest.mark.parametrize("run", [1, 2, 31, 33, 47, 48, 49, 64, 65])
@pytest.mark.parametrize("step", [0, 1, 3])
def test_runs_of_records_in_one_cell_of_the_sort_key(run, step):
    """Bursts whose records share the sorted bits of the key, before and beyond the length that is
    ranked in place, told apart by the bits below (step 3), by the records (0: equal starts) or by
    both, in a window long enough for coarse cells; bursts cross tiles of 256 at every offset."""
    bursts = 700 // run + 40
    at = T0 + np.repeat(np.sort(np.random.default_rng(run).choice(10**6, bursts, replace=False)) * 30_000, run)
    starts = at + np.tile(np.arange(run) * step, bursts)
    ev = _device(len(starts), starts, 5 + np.tile(np.arange(run) % 3, bursts), stream=np.arange(len(starts)) % 2)
    ev = ev[np.random.default_rng(7).permutation(len(ev))]
    for windows in (1, 2):
        off = [0, len(ev)] if windows == 1 else [0, len(ev) // 3, len(ev)]
        both(ev, off, [T0] * windows, [T0 + 31 * 10**9] * windows)


@pytest.mark.parametrize("lanes", [1, 900])
def test_keys_that_fill_their_word(lanes):
    """A window as long as one may be, with enough lanes and records that the key has no room for all time bits
    below the sorted ones: bursts told apart by those it has, by those it has not, and by the records."""
    rng = np.random.default_rng(lanes)
    n = 40_000
    at = rng.integers(0, 1 << 20, n // 8) << 19
    start = T0 + (at[:, None] + rng.integers(0, 4, (n // 8, 8)) * rng.choice([0, 1, 3, 64, 4000], (n // 8, 1))).reshape(-1)
    ev = _device(n, start, rng.integers(0, 3, n), pid=np.repeat(rng.integers(0, lanes, n // 8), 8), kind=2)
    both(ev[rng.permutation(n)], [0, n], [T0], [T0 + (1 << 40) - 1])


def test_one_lane_whose_key_is_all_time_and_index():
    """2^23 records and more of one thread in the longest window: 40 bits of time and 24 of the index."""
    import torch
    from paper_2609_40247_b200 import ta
    n = (1 << 23) + 77
    rng = np.random.default_rng(0)
    ev = np.zeros(n, dtype=EVENT_DTYPE)
    ev["ts_start"] = T0 + np.sort(rng.integers(0, 1 << 39, n)) + (1 << 38)
    ev["ts_end"] = ev["ts_start"] + 1 + np.arange(n) % 3
    ev["corr_id"], ev["kind"] = 1000 - np.arange(n), 2
    ev = ev[np.concatenate([np.arange(i, n, 64) for i in range(64)])]
    buf = torch.from_numpy(ev.view(np.uint8).reshape(-1)).cuda()
    with ta.Window(buf, [0, n], [T0], [T0 + (1 << 40) - 1]) as w:
        s = w.sort_timeline()
        want = np.lexsort((np.arange(n), -ev["ts_end"], ev["ts_start"]))
        assert np.array_equal(s.numpy("perm"), want) and s.n_lanes == 1
        j = w.correlate_launches()
        assert int(j.join_sum["n_launch"][0]) == int(j.join_sum["n_orphan_launch"][0]) == n


@pytest.mark.parametrize("lanes,per", [(1, 3), (2, 255), (257, 9), (1030, 3), (40, 700)])
def test_lane_table_from_the_counts_of_the_load(lanes, per):
    """Lanes of one window from the records counted per triple: one to several rounds of the CTA that
    makes the table, host and device lanes in any order, some records dropped."""
    rng = np.random.default_rng(lanes)
    n = lanes * per
    ev = np.zeros(n, dtype=EVENT_DTYPE)
    lane = rng.permutation(np.arange(n) % lanes)
    ev["pid"] = lane // 5 - lanes // 10
    ev["stream"] = lane % 5
    ev["kind"] = np.where(lane % 5 < 2, 1, 3)
    ev["ts_start"] = T0 + rng.integers(0, 10**9, n)
    ev["ts_end"] = ev["ts_start"] + rng.integers(1, 10**5, n)
    ev["corr_id"] = np.arange(n)
    both(ev, [0, n], [T0], [T0 + 10**9])
    ev["kind"][::11] = 7
    both(ev, [0, n], [T0], [T0 + 10**9])


def test_gather_takes_the_lanes_of_large_processes_together():
    """One process with more records than the gather's order of tiles begins at: two lanes of very
    different lengths and a dropped tail that begins inside a tile."""
    n = 2_700_001
    rng = np.random.default_rng(3)
    ev = np.zeros(n, dtype=EVENT_DTYPE)
    device = np.arange(n) % 7 > 2
    ev["kind"] = np.where(device, 3, 2)
    ev["stream"] = np.where(device, np.where(np.arange(n) % 5000 == 4, 9, 1), 0)
    ev["ts_start"] = T0 + np.arange(n) * 5000 + rng.integers(0, 5000, n)
    ev["ts_end"] = ev["ts_start"] + 2000
    ev["corr_id"] = np.arange(n) // 2
    ev = ev[np.argsort(np.arange(n) // 4096 * 2 + device, kind="stable")]
    ev["kind"][5::4001] = 7
    both(ev, [0, n], [T0], [T0 + n * 5000], min_gap=50_000_000)


@pytest.mark.parametrize("value", [0, 63, 64, 65, 131_071, 131_072, (1 << 26) - 1, 1 << 26, (1 << 32) - 1, 1 << 32, 1 << 36])
@pytest.mark.parametrize("names", [1, 513, 3000])
def test_aggregates_of_values_on_and_off_chip(value, names):
    """Durations around the bins and the word a CTA keeps on chip, mixed with ordinary ones, for as many
    symbols as it has rows and more."""
    rng = np.random.default_rng(value % 1000 + names)
    n = 9000
    dur = np.where(rng.random(n) < 0.3, value, rng.integers(500, 10**6, n))
    ev = _device(n, T0 + np.arange(n) * 1000, dur, name=rng.integers(0, names, n))
    both(ev, [0, n], [T0], [T0 + 10**9])


@pytest.mark.parametrize("names", [1, 5, 31, 33, 300])
def test_aggregates_of_values_of_every_size(names):
    """Durations from nothing to minutes, so that most bins are in none of the slots a CTA keeps and more symbols
    than it has room for have values beyond its words."""
    rng = np.random.default_rng(names)
    n = 30_000
    dur = (2.0 ** rng.uniform(0, 37, n)).astype(np.int64) - 1
    ev = _device(n, T0 + np.arange(n) * 1000, dur, name=rng.integers(0, names, n))
    both(ev, [0, n], [T0], [T0 + 10**9], agg_masks=(56, 8))


def test_aggregate_of_records_of_no_length_takes_no_longer():
    """Values outside the bins of a slot were added up in memory, at the rows of a few symbols: 30 times as long."""
    import torch
    from paper_2609_40247_b200 import ta
    n = 4_000_000
    rng = np.random.default_rng(2)
    times = {}
    for label, dur in (("ordinary", rng.integers(1000, 10**6, n)), ("none", 0), ("one in twenty long", np.where(rng.random(n) < 0.05, 10**8, 9000))):
        ev = _device(n, T0 + np.arange(n) * 5000, dur, name=np.arange(n) % 4)
        ev["corr_id"] = -1
        buf = torch.from_numpy(ev.view(np.uint8).reshape(-1)).cuda()
        with ta.Window(buf, [0, n], [T0], [T0 + 30 * 10**9]) as w:
            w.sort_timeline()
            best = float("inf")
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                w.aggregate_ops(ta.DEVICE_KINDS, 0)
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b))
        times[label] = best
    assert times["none"] < 4 * times["ordinary"] and times["one in twenty long"] < 4 * times["ordinary"], times


@pytest.mark.parametrize("pids,seqs,gap", [(2, 40, 1), (2, 20_000, 1), (64, 30, 1), (65, 30, 1), (8, 900, 1), (8, 50, 1000), (3, 1, 1)])
@pytest.mark.parametrize("windows", [1, 3])
def test_collectives_addressed_and_sorted(pids, seqs, gap, windows):
    """Groups in a table of cells (dense numbers, up to 64 processes) and by sorting (sparse numbers, more
    processes), with processes that take part twice or not at all, ties of the last arrival, a communicator
    of unknown size."""
    rng = np.random.default_rng(pids * 1000 + seqs + windows)
    parts, off = [], [0]
    for w in range(windows):
        rows = []
        for c in range(3):
            for q in range(seqs):
                t = T0 + w * 10**10 + (q * 3 + c) * 10**5
                end = t + 90_000 + int(rng.integers(0, 100))
                for p in range(pids):
                    if rng.random() < 0.02:
                        continue
                    for _ in range(1 + (rng.random() < 0.02)):
                        rows.append(("COLL", p - 1, 7, t + int(rng.integers(0, 4)) * 1000, end, 1000 + c, 5, q * gap - 3))
        ev = make_events(rows)
        parts.append(ev[rng.permutation(len(ev))])
        off.append(off[-1] + len(ev))
    both(np.concatenate(parts), off, [T0 + w * 10**10 for w in range(windows)],
         [T0 + w * 10**10 + 5 * 10**9 for w in range(windows)], comm_sizes=[(1000, pids), (1001, pids + 1)])


@pytest.mark.parametrize("pids,gap", [(1, 1), (1, 2), (2, 3), (8, 1), (8, 9), (4, 100)])
def test_collectives_take_no_more_memory_by_cells_than_by_sorting(pids, gap):
    """Nothing but collectives, so that the handle's pool has no room for the cells: from one cell per group and
    eight members to two cells per member, and to numbers too sparse for cells."""
    import torch
    from paper_2609_40247_b200 import ta
    n = 160_000
    k = np.arange(n)
    ev = _device(n, T0 + k // pids * 500 + k % 7, 100, pid=k % pids, kind=5)
    ev["corr_id"], ev["seq"] = 3, k // pids * gap
    both(ev, [0, n], [T0], [T0 + 10**9], comm_sizes=[(3, pids)])
    buf = torch.from_numpy(ev.view(np.uint8).reshape(-1)).cuda()
    dev, stream = buf.device.index, torch.cuda.current_stream().cuda_stream
    asked = []

    def alloc(nbytes):
        asked.append(nbytes)
        return torch.cuda.caching_allocator_alloc(nbytes, dev, stream)

    with ta.Window(buf, [0, n], [T0], [T0 + 10**9], alloc_fn=alloc, release_fn=torch.cuda.caching_allocator_delete) as w:
        w.sort_timeline()
        del asked[:]
        w.match_collectives([(3, pids)])
    # sorting: waits 8, list 4, keys 24, indices and groups 20, rows 60; and descriptors
    assert sum(asked) <= 120 * n + (1 << 20), asked


@pytest.mark.parametrize("lanes", [1, 2, 15, 16, 17, 33])
@pytest.mark.parametrize("spread", [20, 10**6, 1 << 31])
def test_overlap_of_merged_and_of_sorted_lanes(lanes, spread):
    """Streams of a process merged (up to sixteen) and sorted: many equal starts, rows of 32 records that
    span more than 2^32 ns, lanes of one record beside long ones, two processes and two windows."""
    rng = np.random.default_rng(lanes * 7 + spread % 97)
    parts, off = [], [0]
    for w in range(2):
        ev = []
        for pid in (1, 2):
            for s in range(lanes):
                n = int(rng.integers(1, 4)) if s % 3 == 1 else int(rng.integers(100, 400))
                starts = T0 + np.minimum(np.sort(rng.integers(0, max(1, spread * 100), n)), (1 << 38) - 1)
                ev.append(_device(n, starts, rng.integers(0, spread * 3, n), pid=pid, stream=s, kind=rng.integers(3, 6, n)))
        ev = np.concatenate(ev)
        parts.append(ev[rng.permutation(len(ev))])
        off.append(off[-1] + len(ev))
    both(np.concatenate(parts), off, [T0] * 2, [T0 + (1 << 38)] * 2)


@pytest.mark.parametrize("lanes", [2, 3, 11, 12, 13])
@pytest.mark.parametrize("filling", ["around a cut", "in step", "in turns", "one sparse", "one early"])
def test_overlap_of_lanes_of_any_filling(lanes, filling):
    """Lanes of a process as long as the parts they are merged in (one record less, one more), all at the same
    times, one after the other, and a few records spread over or in front of full lanes; two processes."""
    rng = np.random.default_rng(lanes)
    parts = []
    for pid in (1, 2):
        for s in range(lanes):
            n = {"around a cut": (255, 256, 257, 511, 513, 1, 0)[(s + pid) % 7], "in step": 1000, "in turns": 4 * 300,
                 "one sparse": 40 if s == 1 else 9000, "one early": 300 if s == 1 else 5000}[filling]
            k = np.arange(n)
            starts = {"around a cut": np.sort(rng.integers(0, 300, n)), "in step": k * 100,
                      "in turns": (k // 300 * lanes + s) * 300 + k % 300, "one sparse": np.sort(rng.integers(0, 10**6, n)),
                      "one early": k // 3 if s == 1 else np.sort(rng.integers(80, 10**6, n))}[filling]
            parts.append(_device(n, T0 + starts, rng.integers(0, 250, n), pid=pid, stream=s, kind=rng.integers(3, 6, n)))
    ev = np.concatenate(parts)
    ev["corr_id"][ev["kind"] == 5] = 7  # one communicator
    both(ev[rng.permutation(len(ev))], [0, len(ev)], [T0], [T0 + 10**9])


@pytest.mark.parametrize("pids,windows", [(90, 1), (1300, 4)])
def test_overlap_of_many_lanes_of_one_record(pids, windows):
    """Processes of a host lane and two streams of one or two records: merged where their cuts are few, sorted
    where the table of cuts would be larger than what sorting takes."""
    pid, window = np.tile(np.arange(pids), windows), np.repeat(np.arange(windows), pids)
    t = T0 + window * 10**6
    ev = np.concatenate([_device(len(t), t + 5 + s * 3 + pid % 7, 4 + pid % 5, pid=pid, stream=s, kind=kind)
                         for s, kind in ((0, 1), (0, 3), (1, 4), (1, 3))])
    ev = ev[np.argsort(np.tile(window, 4), kind="stable")]
    both(ev, np.arange(windows + 1) * pids * 4, T0 + np.arange(windows) * 10**6, T0 + np.arange(1, windows + 1) * 10**6)


@pytest.mark.parametrize("shape", ["sparse beside full", "short lanes"])
def test_overlap_takes_no_longer_on_lanes_of_another_filling(shape):
    """300 records spread over 2 M others (with the sparse lane walked record by record through the full one the
    call took 60 times what it takes of two even lanes) and 2000 windows of 64 lanes of eight records (ten
    times, merged): both take about what two even lanes of as many records take."""
    import torch
    from paper_2609_40247_b200 import ta
    rng = np.random.default_rng(5)

    def even(n):
        return [(np.concatenate([_device(n // 2, T0 + np.sort(rng.integers(0, 30 * 10**9, n // 2)), 1000, stream=s)
                                 for s in (0, 1)]), 1)]
    if shape == "short lanes":
        k = np.arange(1 << 20)
        odd = [(_device(len(k), T0 + k // 512 * 10**6 + k % 512 * 1000, 700, pid=k // 64 % 8 * 3, stream=k % 8), 2048)]
        host = _device(2048 * 8, T0 + np.arange(2048 * 8) // 8 * 10**6, 10, pid=np.arange(2048 * 8) % 8 * 3, kind=1)
        odd = [(np.concatenate([odd[0][0], host]), 2048)]
    else:
        odd = [(np.concatenate([_device(n, T0 + np.sort(rng.integers(0, 30 * 10**9, n)), 1000, stream=s)
                                for s, n in enumerate((2_000_000, 300))]), 1)]
    times = []
    for ev, windows in odd + even(len(odd[0][0])):
        window = (ev["ts_start"] - T0) // 10**6 if windows > 1 else np.zeros(len(ev), dtype=np.int64)
        ev = ev[np.argsort(window, kind="stable")]
        off = np.concatenate([[0], np.cumsum(np.bincount(window, minlength=windows))])
        span = 10**6 if windows > 1 else 30 * 10**9
        buf = torch.from_numpy(ev.view(np.uint8).reshape(-1)).cuda()
        with ta.Window(buf, off, T0 + np.arange(windows) * span, T0 + np.arange(1, windows + 1) * span) as w:
            w.sort_timeline()
            best = float("inf")
            for _ in range(8):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                w.device_overlap()
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[0] < 5 * times[1], times


@pytest.mark.parametrize("n", [8192, 262_143, 262_145, 300_000])
def test_long_gaps_ordered_by_one_cta_and_by_many(n):
    """Lists and bitmaps around the size one CTA puts in order: every record behind a long gap, and one
    in ninety."""
    for every in (1, 90):
        wait = np.where(np.arange(n) % every == 0, 700, 0)
        starts = T0 + np.cumsum(wait + 10)
        ev = _device(n, starts, 10, stream=np.arange(n) % 3)
        both(ev, [0, n], [T0], [T0 + (1 << 35)], min_gap=500 if every > 1 else 1)


@pytest.mark.parametrize("n,every", [(8191, 1), (8192, 1), (262_144, 400), (262_145, 400)])
def test_long_gaps_at_the_limits_of_one_cta(n, every):
    """A list of 8192 entries and one more (a gap in front of every record and one behind the last), and a
    bitmap of 8192 words and one more with a list far below."""
    wait = np.where(np.arange(n) % every == 0, 700, 0)
    _, g = both(_device(n, T0 + np.cumsum(wait + 10), 10), [0, n], [T0], [T0 + (1 << 35)], min_gap=500)
    assert len(g["long_gaps"]) == (n + every - 1) // every + 1


@pytest.mark.parametrize("comms", [31, 32, 33, 64])
def test_collectives_of_communicators_few_and_many(comms):
    """Communicator sizes that travel with the launch, and those that are copied: right, too small, not given."""
    rng = np.random.default_rng(comms)
    seqs, pids = 20, 3
    k = np.arange(comms * seqs * pids)
    ev = _device(len(k), T0 + k * 50 + rng.integers(0, 500, len(k)), 40, pid=k % pids, kind=5)
    ev["corr_id"], ev["seq"] = 10**12 - k // pids % comms * 7, k // (pids * comms)
    ev = ev[rng.permutation(len(ev))[:-5]]
    sizes = [(10**12 - c * 7, pids + (c % 5 == 2)) for c in range(comms) if c % 4 != 3]
    both(ev, [0, len(ev)], [T0], [T0 + 10**9], comm_sizes=sizes)


@pytest.mark.parametrize("windows", [1, 2])
@pytest.mark.parametrize("beyond", [0, 1])
def test_collectives_at_the_limit_of_the_cells(beyond, windows):
    """As many cells as two per member and 4096, and one per window more."""
    m = 600 * windows
    last = (2 * m + 4096) // windows - 1 + beyond  # largest sequence number: last + 1 cells a window
    k = np.arange(600)
    one = _device(600, k // 2 * 300, 100, pid=k % 2, kind=5)
    one["corr_id"], one["seq"] = 9, np.where(k // 2 == 299, last, k // 2 * 3)
    parts = []
    for w in range(windows):
        parts.append(one.copy())
        parts[-1]["ts_start"] += T0 + w * 10**6
        parts[-1]["ts_end"] += T0 + w * 10**6
    both(np.concatenate(parts), np.arange(windows + 1) * 600, T0 + np.arange(windows) * 10**6,
         T0 + np.arange(1, windows + 1) * 10**6, comm_sizes=[(9, 2)])


@pytest.mark.parametrize("run", [1, 200])
def test_gather_order_of_processes_of_uneven_size(run):
    """Two processes of 4.9 M and 0.2 M records, whose lanes are taken by turns, one of them without records in the
    first half; with a run of equal times too long to be ranked in place (200) the order is not used."""
    n = 5_100_001
    rng = np.random.default_rng(run)
    k = np.arange(n)
    ev = np.zeros(n, dtype=EVENT_DTYPE)
    ev["pid"] = np.where(k % 25 == 3, 4, 2)
    device = k % 7 > 2
    ev["kind"] = np.where(device, 3, 2)
    ev["stream"] = np.where(device, np.where((k % 5 == 4) & (k > n // 2), 9, 1), 0)
    ev["ts_start"] = T0 + k * 5000 + rng.integers(0, 5000, n)
    ev["ts_start"][1000:1000 + run] = T0 + 7
    ev["ts_end"] = ev["ts_start"] + 2000
    ev["corr_id"] = k // 2
    ev = ev[np.argsort(k // 4096 * 2 + device, kind="stable")]
    both(ev, [0, n], [T0], [T0 + n * 5000], min_gap=50_000_000)


def test_noalloc_call_that_fails_leaves_nothing_to_the_next():
    """A call under stream capture is refused when it comes to wait, after it has taken its place among the
    calls; what follows clears the sums itself."""
    import torch
    from paper_2609_40247_b200 import ta
    start = torch.arange(5000, dtype=torch.int64, device="cuda") * 100 + T0
    end = start + 60
    gap, lane = torch.empty_like(start), torch.zeros(ta.LANE_GAPS.itemsize, dtype=torch.uint8, device="cuda")

    def check():
        _, row = ta.lane_gaps_noalloc(start, end, T0, T0 + 10**6, gap, lane)
        assert int(row["busy"]) == 300_000 and int(row["n_gaps"]) == 5000 and int(row["n_events"]) == 5000
        assert int(gap.sum()) == 4999 * 40

    check()
    check()
    for _ in range(3):
        graph, refused = torch.cuda.CUDAGraph(), False
        try:
            with torch.cuda.graph(graph):
                try:
                    ta.lane_gaps_noalloc(start, end, T0, T0 + 10**6, gap, lane)
                except ta.TaError:
                    refused = True
        except RuntimeError:
            pass  # the capture ends with the error
        assert refused
        torch.cuda.synchronize()
        check()
    check()


@pytest.mark.parametrize("order", ["aaaa", "adad", "ddaa", "aeda"])
def test_noalloc_calls_that_follow_one_another(order):
    """The sums of a call are cleared by the one in front of it: lanes that end their records in
    ascending order (a) and that do not (d: the scan runs too), refused calls between them (e), of
    different sizes."""
    import torch
    from paper_2609_40247_b200 import ta
    rng = np.random.default_rng(11)
    for i, kind in enumerate(order * 2):
        n = (1, 1023, 1025, 70_001)[(i + len(order)) % 4]
        start = T0 + np.cumsum(rng.integers(1, 1000, n))
        end = start + (rng.integers(0, 300, n) if kind == "a" else 0)
        if kind == "a":
            end = np.maximum.accumulate(end)
        elif n > 1:
            end[n // 2] += 10**6
        if kind == "e":
            with pytest.raises(ta.TaError):
                ta.lane_gaps_noalloc(torch.zeros(3, dtype=torch.int64, device="cuda"),
                                     torch.zeros(3, dtype=torch.int64, device="cuda"), 5, 5)
            continue
        t1 = int(end.max()) + 12345
        gap, row = ta.lane_gaps_noalloc(torch.from_numpy(start).cuda(), torch.from_numpy(end).cuda(), T0, t1)
        before = np.concatenate([[T0], np.maximum.accumulate(end)[:-1]])
        want = np.maximum(start - before, 0)
        tail = t1 - int(end.max())
        assert np.array_equal(gap.cpu().numpy(), want)
        assert int(row["idle"]) == int(want.sum()) + tail and int(row["n_events"]) == n
        assert int(row["busy"]) == int(np.maximum(end - np.maximum(start, before), 0).sum())
        assert int(row["n_gaps"]) == int((want > 0).sum()) + 1 and int(row["last_end"]) == int(end.max())
        assert int(row["max_gap"]) == max(int(want.max()), tail) and int(row["first_start"]) == int(start[0])


@pytest.mark.parametrize("n", [255, 257, 1023, 1025, 262_144, 262_145])
def test_gaps_charged_to_operators_by_tiles_of_either_size(n):
    """Operators four deep on two threads of one process, beside a process without streams and one with
    nothing but streams: around the smaller tile, the larger one and the line between them."""
    rng = np.random.default_rng(n)
    k = np.arange(n)
    ev = np.zeros(n, dtype=EVENT_DTYPE)
    device = k % 5 > 2
    ev["pid"] = np.where(k % 97 == 3, 2, np.where(k % 97 == 1, 1, 0))
    device = np.where(ev["pid"] == 1, False, np.where(ev["pid"] == 2, True, device))
    ev["stream"] = np.where(device, k // 5 % 7, k // 3 % 2)
    ev["kind"] = np.where(device, 3, 2)
    ev["ts_start"] = T0 + 100 + k * 20
    ev["ts_end"] = ev["ts_start"] + np.where(device, rng.integers(1, 60, n), 10)
    ev["corr_id"] = k
    for pid in (0, 1):
        for thread in (0, 1):
            at = k[~device & (ev["pid"] == pid) & (ev["stream"] == thread)]
            for level, every in enumerate((7200, 720, 36, 9)):
                if len(at) < 2:
                    continue
                first = np.arange(0, len(at), every)  # of every block, one record later per level
                last = np.minimum(first + every, len(at)) - 1
                head = np.minimum(first + level, last)
                ev["kind"][at[head]] = 0
                ev["ts_end"][at[head]] = T0 + 100 + at[last] * 20 + 18 - 2 * level
    both(ev[rng.permutation(n)], [0, n], [T0], [T0 + 10**9], min_gap=30)
